// fft_uneven.cuh -- the line pass of batched uneven lengths (fb_fft_plan_many):
// single-pass lines, four-step columns and four-step rows of any 5-smooth
// length up to 2048, power-of-two or not.  k_fft_uneven runs every pass of
// one phase of such a batch in one launch (phase 0: single passes and
// columns; phase 1: rows); k_fft_uneven_one (below) runs both phases in ONE
// launch, each row chunk after its columns.
//
// Jobs (one UnevenDesc per length group or four-step chunk, each with its own
// offset tables, strides, radix schedule and twiddle tables) sit in a device
// table; a device prefix table gives each job's first global tile.
// k_fft_uneven's persistent CTAs walk the global tiles blockIdx.x,
// +gridDim.x, ... (k_fft_uneven_one's claim them from a counter).
//
// A tile runs as in fft_mr.cuh, with the job's shape read from its descriptor:
// stages of composite radices up to 16 (two for most lengths up to 256, three
// above), loads straight from global memory into registers, exchanges through
// one or two shared-memory buffers, stores straight back.  A control warp beside
// the eight compute warps walks the job table one tile ahead.
//
// What bounds it: latency (issue slots 36 % busy; per issue 5.8 warps wait for
// global loads, 4.0 at barriers; 72 registers leave three CTAs per SM).  On 4096
// lengths in [64, 65536] the large radices and the control warp more than halved the
// instructions (417 -> 188 M warp instructions, 166 -> 75 thread instructions per
// value and pass): the radices took 565 -> 530 us, the table walk, claims and
// counter traffic on the control warp 530 -> 418 us.  256 waiting requests of a
// server, 2190 -> 1650 us: there the strided tiles of 1000- to 2048-point lines
// (rows of 2 to 4 values) take most of the time.  Measured without gain: 128
// compute threads and 2048 values per tile (420 us; the server's long lines then
// have rows of 1 or 2: 2110), tiles claimed in pairs (434), twiddles read ahead of
// each stage's barrier (417).
#pragma once

#include <algorithm>

#include "fft_device.cuh"
#include "fft_mr.cuh"

namespace fbfft {

constexpr int kUnevenThreads = 256;
constexpr int kUnevenCtas = 3;        // per SM: 72 registers, 70 KB of exchange buffers
constexpr int kUnevenCap = 4096;      // values per tile
// ... and of a server launch whose tiles would not even give every SM one: twice as
// many SMs work then.  Lone requests, us on the device with tiles of 4096 / 2048 /
// 1024 values: 512 x 512 22.3 / 18.7 / 18.5, 2^18 22.7 / 19.1 / 19.4, 256 x 256 19.0 /
// 16.0 / 15.8, 16384 16.7 / 15.3 / 15.2; once there is a tile for every SM the wide ones
// win (8 requests of 2^19: 69 against 80 us).
constexpr int kUnevenNarrowCap = 2048;
constexpr int kUnevenMaxLen = 2048;   // longest line of a job
constexpr int kUnevenMaxRadix = 16;
constexpr int kUnevenMaxLines = 128;  // contiguous lines per tile

// Kernel argument: the job table and the tile prefix table (device memory,
// written once when the plan is built, or per launch by the request server)
// and the buffers of this exec.  A job's `in` / `out` fields hold element
// offsets into the buffer its in_buf / out_buf names, or (kind 3) addresses.
struct UnevenArgs {
    const UnevenDesc* jobs;   // [njobs]
    const int* tile_start;  // [njobs + 1]: first global tile of each job; [njobs] = all tiles
    const float2* in;       // buffer 0: the caller's input
    float2* out;            // buffer 1: the caller's output
    float2* scratch;        // buffer 2: the plan's four-step intermediate
    int njobs;
    int scale_on;           // 1: jobs marked apply_scale multiply by their `scale`
    // One-launch form (k_fft_uneven_one) only: device counters, nsync of
    // them, zero between execs -- [0] tiles claimed, [1] CTAs finished,
    // [1 + s] finished tiles of dependency slot s >= 1 (UnevenDesc::dep_post /
    // dep), [nsync - 1] finished column tiles of the batch.
    unsigned long long* sync;
    int nsync;
    int columns;            // column tiles of the batch
    int dep_extra;          // test hook: added to every dependency target (the waits then run out)
};

// Kernel argument of the inline form: the tables themselves (a.jobs and
// a.tile_start unused).  About 7.6 KB, well under the 32 KB parameter limit.
constexpr int kUnevenInlineJobs = 16;
struct UnevenInlineArgs {
    UnevenArgs a;
    UnevenDesc jobs[kUnevenInlineJobs];
    int tile_start[kUnevenInlineJobs + 1];
};

#ifdef __CUDACC__

// Tile t of job d: outer index o, first line c0, valid lines Tv (32-bit: a
// job has fewer than 2^31 tiles and lines).
struct UTileIdx {
    int o, c0, Tv;
};
__device__ __forceinline__ UTileIdx utile_index(const UnevenDesc& d, int tile)
{
    UTileIdx ti;
    const int tpo = (int)d.tiles_per_o;
    ti.o = (int)((unsigned)tile / (unsigned)tpo);
    ti.c0 = (tile - ti.o * tpo) * d.T;
    const int rem = (int)d.C - ti.c0;
    ti.Tv = rem < d.T ? rem : d.T;
    return ti;
}

// A job's input / output base in this exec's buffers; kind 3: the field is
// the address itself (jobs of different requests in one server launch).
__device__ __forceinline__ const float2* ubuf_in(const UnevenArgs& a, const UnevenDesc& d)
{
    if (d.in_buf == 3) return d.in;
    const float2* b = d.in_buf == 0 ? a.in : (d.in_buf == 1 ? a.out : a.scratch);
    return b + (long long)reinterpret_cast<uintptr_t>(d.in);
}
__device__ __forceinline__ float2* ubuf_out(const UnevenArgs& a, const UnevenDesc& d)
{
    if (d.out_buf == 3) return d.out;
    float2* b = d.out_buf == 1 ? a.out : a.scratch;
    return b + (long long)reinterpret_cast<uintptr_t>(d.out);
}
// Global start of line (o, c) of the input / output (offset tables or strides).
__device__ __forceinline__ const float2* uline_in(const UnevenArgs& a, const UnevenDesc& d, int o, int c)
{
    const float2* in = ubuf_in(a, d);
    if (d.off_in) return in + (d.in_tfast ? d.off_in[o] + c : d.off_in[c]);
    return in + (long long)o * d.in_so + (long long)c * d.in_sc;
}
__device__ __forceinline__ float2* uline_out(const UnevenArgs& a, const UnevenDesc& d, int o, int c)
{
    float2* out = ubuf_out(a, d);
    if (d.off_out) return out + (d.out_tfast ? d.off_out[o] + c : d.off_out[c]);
    return out + (long long)o * d.out_so + (long long)c * d.out_sc;
}

// A value of the batch: read once per pass, so its line leaves L1 first.
__device__ __forceinline__ float2 uload(const float2* p)
{
    float2 v;
    asm volatile("ld.global.L1::evict_first.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
// What the control warp works out about a tile before the compute warps get
// it: its place (number < 0: no more tiles), its first line's input and
// output, and where its other contiguous lines start relative to that.
struct UTile {
    int number;
    UTileIdx ti;
    const float2* in;
    float2* out;
    long long line[kUnevenMaxLines];
};

// exp(-2 pi i m / N) from the job's two split four-step tables (m < N < 2^31).
__device__ __forceinline__ float2 uptw(const UnevenDesc& d, unsigned m)
{
    return cmul(__ldg(d.ptw_hi + (m >> d.ptw_log)), __ldg(d.ptw_lo + (m & ((1u << d.ptw_log) - 1))));
}

// Stage twiddles w^r, w = w_{Ns R}^k, of a butterfly at position k (table entry
// (r-1) Ns + k): small radices read every factor; from 8 on w and every fourth
// power are read and the others formed by at most three products in a row.
// Every tile reads its own job's tables, which mostly miss L1: few loads, and
// those ahead of the barrier the stage starts with.
template <int R>
struct UTwiddle {
    static constexpr int N = R <= 6 ? (R > 1 ? R - 1 : 1) : 1 + (R - 1) / 4;
    float2 w[N];
    // the power of w that w[m] holds
    __host__ __device__ static constexpr int power(int m) { return R <= 6 ? m + 1 : (m ? 4 * m : 1); }
    __device__ __forceinline__ void load(const float2* tw, int Ns)  // tw: the table at k
    {
        if constexpr (R > 1) {
#pragma unroll
            for (int m = 0; m < N; ++m) w[m] = __ldg(tw + (power(m) - 1) * Ns);
        }
    }
    template <bool FWD>
    __host__ __device__ __forceinline__ void apply(float2* v) const
    {
        if constexpr (R <= 6) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = twmul<FWD>(v[r], w[r - 1]);
        } else {
            const float2 w1 = w[0], w2 = cmul(w1, w1), w3 = cmul(w2, w1);
            v[1] = twmul<FWD>(v[1], w1);
            v[2] = twmul<FWD>(v[2], w2);
            v[3] = twmul<FWD>(v[3], w3);
#pragma unroll
            for (int r = 4; r < R; ++r) {
                const float2 x = w[r / 4];
                v[r] = twmul<FWD>(v[r], r % 4 == 0 ? x : cmul(x, r % 4 == 1 ? w1 : (r % 4 == 2 ? w2 : w3)));
            }
        }
    }
};

// Barrier among the compute warps (named barrier 1).
__device__ __forceinline__ void usync() { asm volatile("bar.sync 1, %0;" ::"n"(kUnevenThreads) : "memory"); }

// One stage of radix R over the tile, lines and positions as in fft_mr.cuh
// with the shape read from the descriptor: the first stage loads its
// butterflies from global memory, stage st >= 1 reads exchange buffer
// (st - 1) & 1, every stage but the last writes buffer st & 1, the last stores
// to global memory with the four-step twiddle and the scale applied.
template <int R, bool FWD, int POS>
__device__ __forceinline__ void ustage(const UnevenArgs& a, const UnevenDesc& d, const UTile& tl, int st, float2* buf)
{
    constexpr bool first = POS == kPosFirst;
    constexpr bool last = POS == kPosLast;
    static_assert(POS == kPosFirst || POS == kPosMid || POS == kPosLast, "stage positions of the uneven kernel");
    const int L = d.L, logT = d.logT, LR = L / R;
    const bool in_tf = d.in_tfast != 0, out_tf = d.out_tfast != 0;
    const bool tf = first ? in_tf : out_tf;
    const int Tv = tl.ti.Tv, nb = tf ? (LR << logT) : Tv * LR;
    const unsigned lrm = d.lr_mag[st];
    const int Ns = first ? 1 : d.ns[st];
    const unsigned nsm = first ? 0u : d.ns_mag[st];
    const float2* twb = d.tw + (first ? 0 : d.twoff[st]);
    const float2* rd = (st & 1) ? buf : buf + d.xbuf;
    float2* wr = (st & 1) ? buf + d.xbuf : buf;
    const int rrow = first ? 0 : d.xrow[st], rpad = first ? 0 : d.xpad[st], rstep = first ? 0 : d.xstep[st];
    const int wrow = last ? 0 : d.xrow[st + 1], wblk = last ? 0 : Ns * R + d.xpad[st + 1];
    const float2* in0 = first ? tl.in : nullptr;
    float2* out0 = last ? tl.out : nullptr;
    const long long sn = first ? (in_tf ? d.in_sn : 1) : (last ? (out_tf ? d.out_sk : 1) : 0);
    const bool ptw = last && d.ptw != 0, scale = last && a.scale_on && d.apply_scale;
    const float sc = scale ? d.scale : 1.0f;
    const int c0 = ptw ? tl.ti.c0 : 0;
    const float2* p4t = ptw ? buf + d.ptw_at : nullptr;
    int b = threadIdx.x, t = 0, j = 0, q = 0, k = 0;
    UTwiddle<R> tw;
    float2 plo = make_float2(0.f, 0.f), phi = plo;
#pragma unroll
    for (int m = 0; m < tw.N; ++m) tw.w[m] = make_float2(0.f, 0.f);
    auto place = [&]() {  // butterfly b: line t, position j = q Ns + k, and its table reads
        if (tf) {
            t = b & ((1 << logT) - 1);
            j = b >> logT;
        } else {
            t = lrm ? (int)__umulhi((unsigned)b, lrm) : b;
            j = b - t * LR;
        }
        if constexpr (last) {
            k = j;  // Ns = L / R
        } else if constexpr (first) {
            q = j;
        } else {
            q = (int)__umulhi((unsigned)j, nsm);
            k = j - q * Ns;
        }
        if constexpr (!first) tw.load(twb + k, Ns);
        if (ptw && t < Tv) {
            const unsigned m = (unsigned)(c0 + t) * (unsigned)j;  // below N: c0 + t < C
            phi = __ldg(d.ptw_hi + (m >> d.ptw_log));
            plo = __ldg(d.ptw_lo + (m & ((1u << d.ptw_log) - 1)));
        }
    };
    if constexpr (!first) usync();
    if (b < nb) place();
    while (b < nb) {
        if (t < Tv) {
        float2 v[R];
        if constexpr (first) {
            const float2* p = in0 + (in_tf ? j * sn + t : tl.line[t] + j);
            const long long step = LR * sn;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = uload(p + r * step);
        } else {
            const float2* p = rd + t * rrow + j + q * rpad;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = p[r * rstep];
            tw.template apply<FWD>(v);
        }
        mr_dft<R, FWD>(v);
        if constexpr (!last) {
            float2* p = wr + t * wrow + q * wblk + k;
#pragma unroll
            for (int r = 0; r < R; ++r) p[r * Ns] = v[r];
        } else {
            // the outputs of butterfly j are j + r Ns
            float2* p = out0 + (out_tf ? j * sn + t : tl.line[t] + j);
            const long long step = Ns * sn;
            if (ptw) {
                // exp(-2 pi i c (j + r Ns) / N): one table product per butterfly
                // times the tile's own factor exp(-2 pi i c r Ns / N)
                const float2 w = cmul(phi, plo);
                const float2* p4 = p4t + t;
                v[0] = twmul<FWD>(v[0], w);
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = twmul<FWD>(v[r], cmul(w, p4[r << logT]));
            }
            if (scale) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = sc * v[r];
            }
#pragma unroll
            for (int r = 0; r < R; ++r) p[r * step] = v[r];
        }
        }
        b += kUnevenThreads;
        if (b < nb) place();
    }
}

// Stage st, any radix of a schedule.
template <bool FWD, int POS>
__device__ __forceinline__ void ustage_any(const UnevenArgs& a, const UnevenDesc& d, const UTile& tl, int st, float2* buf)
{
    switch (d.radix[st]) {
#define FB_USTAGE(R) \
    case R: ustage<R, FWD, POS>(a, d, tl, st, buf); break;
        FB_USTAGE(2)
        FB_USTAGE(3)
        FB_USTAGE(4)
        FB_USTAGE(5)
        FB_USTAGE(6)
        FB_USTAGE(8)
        FB_USTAGE(9)
        FB_USTAGE(10)
        FB_USTAGE(12)
        FB_USTAGE(15)
        FB_USTAGE(16)
#undef FB_USTAGE
    default:  // radix 1: a copy (one-radix schedules)
        ustage<1, FWD, POS>(a, d, tl, st, buf);
        break;
    }
}
// Every stage of tile tl of job d, by the compute warps.
template <bool FWD>
__device__ __forceinline__ void utile_run(const UnevenArgs& a, const UnevenDesc& d, const UTile& tl, float2* buf)
{
    ustage_any<FWD, kPosFirst>(a, d, tl, 0, buf);
    if (d.ptw) {  // four-step columns: the factors of the tile's lines the last stage needs
        const int R = d.radix[d.nst - 1], step = d.ns[d.nst - 1], T = 1 << d.logT;
        for (int e = threadIdx.x; e < (R << d.logT); e += kUnevenThreads)
            if ((e & (T - 1)) < tl.ti.Tv)  // c < C: the product stays below N
                buf[d.ptw_at + e] = uptw(d, (unsigned)(tl.ti.c0 + (e & (T - 1))) * (unsigned)((e >> d.logT) * step));
    }
    const int nst = d.nst;  // each stage from here on starts with a barrier
    for (int s = 1; s < nst - 1; ++s) ustage_any<FWD, kPosMid>(a, d, tl, s, buf);
    ustage_any<FWD, kPosLast>(a, d, tl, nst - 1, buf);
}

// Control warp: ask L2 for the values a tile will read.
__device__ __forceinline__ void uprefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void utile_prefetch(const UnevenDesc& d, const UTile& tl, int lane)
{
    const int Tv = tl.ti.Tv;
    if (d.in_tfast) {
        for (int n = lane; n < d.L; n += 32) {
            const float2* p = tl.in + (long long)n * d.in_sn;
            uprefetch(p);
            if ((((uintptr_t)p ^ (uintptr_t)(p + Tv - 1)) >> 7) != 0) uprefetch(p + Tv - 1);
        }
    } else {
        const int per = (d.L + 15) / 16;  // 128-byte lines of a line of values
        for (int i = lane; i < Tv * per; i += 32) {
            const int t = i / per;
            uprefetch(tl.in + tl.line[t] + (i - t * per) * 16);
        }
    }
}
// Control warp: fill in the tile of job d.
__device__ __forceinline__ void utile_find(const UnevenArgs& a, const UnevenDesc& d, int number, UTile& tl, int lane)
{
    const UTileIdx ti = utile_index(d, number);
    const bool in_c = !d.in_tfast, out_c = !d.out_tfast;
    if (lane == 0) {
        tl.number = number;
        tl.ti = ti;
        tl.in = uline_in(a, d, ti.o, ti.c0);
        tl.out = uline_out(a, d, ti.o, ti.c0);
    }
    if (in_c || out_c) {
        // contiguous lines: a side's offset table, or its line stride (the same
        // on both sides where both are contiguous)
        const long long* off = in_c ? d.off_in : d.off_out;
        const long long sc = in_c ? d.in_sc : d.out_sc;
        for (int t = lane; t < ti.Tv; t += 32)
            tl.line[t] = off ? off[ti.c0 + t] - off[ti.c0] : (long long)t * sc;
    }
}

// A word of the job or tile-prefix table: read-only global memory, or (INL)
// the kernel's own parameter, which takes plain generic loads.
template <bool INL>
__device__ __forceinline__ int utab(const int* p)
{
    if constexpr (INL)
        return *p;
    else
        return __ldg(p);
}

// ---------------------------------------------------------------------------
// The CTA: kUnevenThreads compute threads and one control warp.  The control
// warp walks the tiles one ahead of the compute warps -- it finds the next
// tile's job, copies its descriptor to shared memory, sees to its
// dependencies and asks L2 for its values -- so none of those latencies (about
// ten dependent global accesses a tile) is on the compute warps' path.
// Hand-over by named barriers: ready[b] (control arrives, compute waits) says
// slot b holds a tile whose inputs are there, done[b] (compute arrives, control
// waits) that slot b's tile is finished.  ready[b] also separates the compute
// warps' use of the exchange buffers from one tile to the next.
//
// Tiles are assigned round robin (ONE = false), or (ONE) claimed in table order
// from a device counter, every pass of a batched uneven exec in ONE launch.  The
// job table then holds the single passes and four-step columns, then the
// four-step rows; a row reads what the columns of its chunk wrote, so it may
// start only once they are done.  A claimed tile always belongs to a running
// CTA, so a row tile waits only for column tiles already held by running CTAs,
// and a column tile never waits (a CTA claims in increasing order, so whatever
// it holds before a column tile is a column tile too; a tile's count is
// published before the control warp waits for the next tile's inputs).  No CTA
// can therefore wait on one that is not resident, whatever else shares the GPU.
// A finished column tile raises its chunk's counter: its stores, done[b], then
// a fence and a release add by one control lane (the fence is cumulative over
// what the barrier ordered before it).  A row tile starts once an acquire read
// sees the counter at the chunk's column-tile count; the last column tile of
// the batch is counted in `all`, and once a CTA has seen every column done it
// reads no more counters.  The wait is bounded: past the limit the error word is
// set and the tile runs anyway.  The last CTA to finish zeroes the counters for
// the next exec.
// ---------------------------------------------------------------------------
template <int ID>
__device__ __forceinline__ void ubar_sync()
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(kUnevenThreads + 32) : "memory");
}
template <int ID>
__device__ __forceinline__ void ubar_arrive()
{
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(kUnevenThreads + 32) : "memory");
}
// ready[b]: barriers 2, 3; done[b]: 4, 5.
__device__ __forceinline__ void uready_wait(int b) { b ? ubar_sync<3>() : ubar_sync<2>(); }
__device__ __forceinline__ void uready_post(int b) { b ? ubar_arrive<3>() : ubar_arrive<2>(); }
__device__ __forceinline__ void udone_wait(int b) { b ? ubar_sync<5>() : ubar_sync<4>(); }
__device__ __forceinline__ void udone_post(int b) { b ? ubar_arrive<5>() : ubar_arrive<4>(); }

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add_u64(unsigned long long* p, unsigned long long v)
{
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// One lane: whether column tiles number `need` are counted in slot `dep`.
__device__ __forceinline__ bool udeps_ready(const UnevenArgs& a, int dep, int need)
{
    return ld_acquire_u64(a.sync + 1 + dep) >= (unsigned long long)need + (unsigned long long)a.dep_extra;
}
// The same, waited for at most kWaitLimitNs; past it set the error word.  Once
// the word is set (by any CTA) no wait lasts longer, so a launch whose waits
// cannot end still ends within about one limit.
__device__ __forceinline__ void udeps_wait(const UnevenArgs& a, int dep, int need, int* err)
{
    const unsigned long long t0 = global_ns();
    while (!udeps_ready(a, dep, need)) {
        if (*reinterpret_cast<volatile int*>(err) != 0) return;
        if (global_ns() - t0 > kWaitLimitNs) {
            atomicExch(err, 1);
            return;
        }
        __nanosleep(200);
    }
}

template <bool FWD, bool INL, bool ONE>
__device__ __forceinline__ void uneven_body(const UnevenArgs& a, const UnevenDesc* jobs, const int* tile_start)
{
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    float2* buf = reinterpret_cast<float2*>(smem_dyn);
    __shared__ UnevenDesc sd[2];  // the descriptors of two tiles in turn
    __shared__ UTile s_tile[2];
    pdl_start();
    if (threadIdx.x < kUnevenThreads) {
        for (int b = 0;; b ^= 1) {
            uready_wait(b);
            if (s_tile[b].number < 0) return;
            utile_run<FWD>(a, sd[b], s_tile[b], buf);
            udone_post(b);
        }
    }
    // ---- control warp ----
    const int lane = threadIdx.x & 31;
    const int total = utab<INL>(tile_start + a.njobs);
    int j = 0, g = ONE ? 0 : (int)blockIdx.x;
    int post = 0;           // dependency slot + 1 the running tile raises
    int seen = 0;           // the last dependency slot + 1 found complete
    bool all = false;       // every column tile of the batch is known to be done
    for (int i = 0;; ++i) {
        const int b = i & 1;
        if constexpr (ONE) {
            if (lane == 0) g = (int)atomicAdd(a.sync, 1ull);
            g = __shfl_sync(0xffffffffu, g, 0);
        } else if (i > 0) {
            g += (int)gridDim.x;
        }
        const bool has = g < total;
        int next_post = 0, dep = 0, need = 0;
        if (has) {
            // the job of tile g: 32 entries of the prefix table at a time
            for (;;) {
                const int e = j + 1 + lane;
                const unsigned m = __ballot_sync(0xffffffffu, e <= a.njobs && g >= utab<INL>(tile_start + e));
                j += __popc(m);
                if (m != 0xffffffffu) break;
            }
            const int* src = reinterpret_cast<const int*>(jobs + j);
            int* dst = reinterpret_cast<int*>(&sd[b]);
            for (int w = lane; w < (int)(sizeof(UnevenDesc) / 4); w += 32) dst[w] = utab<INL>(src + w);
            __syncwarp();
            utile_find(a, sd[b], g - utab<INL>(tile_start + j), s_tile[b], lane);
            next_post = sd[b].dep_post;
            if (ONE && !all && sd[b].dep != seen) dep = sd[b].dep, need = sd[b].dep_need;
        } else if (lane == 0) {
            s_tile[b].number = -1;
        }
        bool ready = true;
        if (ONE && dep != 0) {
            unsigned ok = 0;
            if (lane == 0) {
                // every column tile counted (slot 0's own counter): no more reads after this
                ok = udeps_ready(a, dep, need) ? 1u : 0u;
                if (ok && ld_acquire_u64(a.sync + a.nsync - 1) >= (unsigned long long)a.columns + a.dep_extra) ok = 2u;
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            ready = ok != 0;
            all = ok == 2u;
            if (ready) seen = dep;
        }
        __syncwarp();
        if (ready) {
            uready_post(b);
            if (has) utile_prefetch(sd[b], s_tile[b], lane);
        }
        if (i > 0) {
            udone_wait(b ^ 1);
            if (ONE && post && lane == 0) {
                __threadfence();
                red_release_add_u64(a.sync + 1 + post, 1ull);
                red_release_add_u64(a.sync + a.nsync - 1, 1ull);
            }
        }
        if (!ready) {
            if (lane == 0) udeps_wait(a, dep, need, sd[b].err);
            __syncwarp();
            uready_post(b);
        }
        post = next_post;
        if (!has) break;
    }
    if constexpr (ONE) {
        // the last CTA out zeroes the counters (every other CTA's atomics are
        // ordered before its finish count by the fences)
        unsigned last = 0;
        if (lane == 0) {
            __threadfence();
            last = atomicAdd(a.sync + 1, 1ull) == (unsigned long long)gridDim.x - 1 ? 1u : 0u;
            if (last) __threadfence();
        }
        if (__shfl_sync(0xffffffffu, last, 0))
            for (int k = lane; k < a.nsync; k += 32) a.sync[k] = 0ull;
    }
}

constexpr int kUnevenBlock = kUnevenThreads + 32;

template <bool FWD>
__global__ void __launch_bounds__(kUnevenBlock, kUnevenCtas) k_fft_uneven(const __grid_constant__ UnevenArgs a)
{
    uneven_body<FWD, false, false>(a, a.jobs, a.tile_start);
}

template <bool FWD>
__global__ void __launch_bounds__(kUnevenBlock, kUnevenCtas) k_fft_uneven_one(const __grid_constant__ UnevenArgs a)
{
    uneven_body<FWD, false, true>(a, a.jobs, a.tile_start);
}

// The same pass with its job and tile-prefix tables inside the kernel
// parameter (at most kUnevenInlineJobs jobs): a small batch then needs no
// copy of its tables to the device before it can start.
template <bool FWD>
__global__ void __launch_bounds__(kUnevenBlock, kUnevenCtas) k_fft_uneven_inline(const __grid_constant__ UnevenInlineArgs p)
{
    uneven_body<FWD, true, false>(p.a, p.jobs, p.tile_start);
}

#endif  // __CUDACC__

// Host side (fft_kernels_uneven.cu).
cudaError_t uneven_launch(bool forward, const UnevenArgs& a, long long grid, size_t smem, cudaStream_t stream);
cudaError_t uneven_occupancy(bool forward, size_t smem, int* blocks_per_sm);
cudaError_t uneven_launch_inline(bool forward, const UnevenInlineArgs& a, long long grid, size_t smem,
                                 cudaStream_t stream);
cudaError_t uneven_occupancy_inline(bool forward, size_t smem, int* blocks_per_sm);
cudaError_t uneven_launch_one(bool forward, const UnevenArgs& a, long long grid, size_t smem, cudaStream_t stream);
cudaError_t uneven_occupancy_one(bool forward, size_t smem, int* blocks_per_sm);

// Schedules of every line length of the engine, worked out once per process.
inline const MrSchedule& uneven_schedule(int L, bool contiguous)
{
    struct Table {
        MrSchedule s[2][kUnevenMaxLen + 1] = {};
        Table()
        {
            for (int n = 2; n <= kUnevenMaxLen; ++n) {
                int m = n;
                for (int p : {2, 3, 5})
                    while (m % p == 0) m /= p;
                if (m == 1)
                    for (int k = 0; k < 2; ++k) s[k][n] = mr_schedule(n, k != 0, kUnevenMaxRadix);
            }
        }
    };
    static const Table table;
    return table.s[contiguous ? 1 : 0][L];
}

// Lines per tile of a job of L-point lines (C per outer index): as many as fit
// `cap` values -- any number of contiguous lines (at most 128), a power of two
// where a side is strided (rows of T consecutive values: 16, or 32 for short
// lines, whatever fits).
inline int uneven_lines(long long L, long long C, int io, int cap = kUnevenCap)
{
    auto floor2 = [](long long x) {
        long long p = 1;
        while (p * 2 <= x) p *= 2;
        return p;
    };
    long long T = std::max(1LL, cap / L);
    if (io == 0)  // contiguous on both sides
        T = std::min<long long>(std::min<long long>(T, kUnevenMaxLines), C);
    else
        T = std::min(std::min(floor2(T), L <= 64 ? 32LL : 16LL), C <= 1 ? 1LL : 2 * floor2(C - 1));
    return (int)std::max(1LL, T);
}

// Shape of such a job on the one-kernel batched-uneven engine: the
// composite-radix schedule of radices up to 16, and uneven_lines per tile.
inline MrConfig uneven_shape(long long L, long long C, int io, int cap = kUnevenCap)
{
    MrConfig c{};
    c.L = (int)L, c.io = io;
    const MrSchedule& s = uneven_schedule((int)L, io == 0);
    c.n = L == 1 ? 2 : s.n;  // one point: two copies
    for (int i = 0, ns = 1; i < c.n; ++i) {
        c.radix[i] = L == 1 ? 1 : s.radix[i];
        c.ns[i] = ns;
        ns *= c.radix[i];
    }
    c.T = uneven_lines(L, C, io, cap);
    return c;
}

// Row placement rules for tiles of a power of two of lines whose rows are not
// padded inside.  No kernel's tiles are laid out by these two any more (mr_place
// finds every job's rows); the host index test still checks them.
// Row stride (elements) of a tile's work rows: at least L, and chosen so that the
// 16 threads of a half-warp never meet on one bank of 8-byte words across rows.
// A stage that maps consecutive threads to consecutive lines (the strided sides
// of four-step jobs) puts H = 16/T positions of each of T lines in a half-warp; a
// stage that maps them along a line puts H = G = 256/T positions of each of 16/G
// lines there (short lines, G < 16).  Rows then start H * (odd) banks apart when
// stride mod 2H == H.  (A tile of 32 strided lines has both kinds of stage; its
// lines-fast stages win: H = 1.)
inline int uneven_line_stride(long long L, long long T, bool cfast)
{
    const long long G = kUnevenThreads / T;
    long long H = 1;
    if (cfast && T <= 16) H = 16 / T;
    else if (!cfast && G < 16) H = G;
    long long ls = L;
    if (H < 16)
        while (ls % (2 * H) != H) ++ls;
    return (int)ls;
}

// Row stride of a contiguous-input tile copied to shared memory before its first
// stage (0: rows of L, first stage along a line).  Tiles of 2 to 8 lines land in
// rows H = 16/T banks apart (stride mod 2H == H, even, so the 16-byte copies stay
// aligned) and their first stage maps threads across lines: its radix-R groups
// would otherwise fill a half-warp at stride R (8-way for radix 8).
inline int uneven_land_row(long long L, long long T, bool in_tfast)
{
    if (in_tfast || T < 2 || T > 8) return 0;
    const long long H = 16 / T;
    long long lr = L;
    while (lr % (2 * H) != H) ++lr;
    return (int)lr;
}

}  // namespace fbfft

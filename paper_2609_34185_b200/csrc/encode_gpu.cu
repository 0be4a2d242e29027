// CUDA back end of the EntroPack encoder (paper Sec. 3.2-3.6): row RMS, E8 quantisation with field
// histograms, the bisection of Algorithm 1, the rate correction, row-scale refit and tiled 32-state rANS encoding run on the
// GPU, one stream of launches without a wait in between.  The final tables are made there, for coding, and on the host, for the
// blob, from the same counts (a few kilobytes) by the code of the host back end, which compares the two; that also takes over a search
// whose decisions the device leaves open.  Both back ends produce the same bytes for the same input.
//
// Every result that enters the stream is the host code's bit for bit.  Where the host's operation order is
// expensive here (two divisions per weight, sums in index order), the kernel computes the value another way together
// with a bound on the difference, keeps it if no value inside the bound would round or compare differently, and
// otherwise repeats the host's operations.
#include <cuda_runtime.h>

#include <mutex>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <new>
#include <vector>

#include "encoder_core.hpp"

namespace ep {
int check_encode_args(uint32_t R, uint32_t C, double target_bpp, const ep_encode_opts &o);
}

namespace {

using namespace ep;

constexpr int kHistOrigin = -4096;       // kHistBins values per table: -4096 .. 4095
constexpr uint32_t kMaxTableSymbols = 40960;   // sum of K over the 17 tables that a stream of this back end may have
constexpr uint32_t kFewEntries = 2048, kSmemEntries = 11264;   // tile coder: entries in shared memory with several CTAs per SM, with one
constexpr double kUnit = 1.1102230246251565e-16;   // 2^-53, the rounding unit of double

// the wait of a kernel that is launched while the one before it ends (launch_chained): before it, only kernel parameters are read
__device__ __forceinline__ void chained_start() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// All threads of a CTA: is it the last of `n` CTAs to get here?  What the others did before they got here is there for the last one.
// One thread's fences next to the atomic order the whole CTA's accesses (a barrier orders them within the CTA, and fences are
// cumulative).  With a fence in each of 1024 threads the six passes of 512 x 1024 at 4 bpp, first to last, took 98.6 us, 96.4 so.
__device__ __forceinline__ bool arrive_last(uint32_t *counter, uint32_t n, uint32_t &shared_flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        shared_flag = atomicAdd(counter, 1u) == n - 1u;
        __threadfence();
    }
    __syncthreads();
    return shared_flag != 0;
}

// ---- sums over a row ------------------------------------------------------------------------------------
// The row RMS (Sec. 3.2) and Eq. 13 are defined by sums in double in index order, a chain of dependent additions per
// row (14 cycles each: 60 us for 8192 of them, whatever the bandwidth).  Here a CTA sums a row in parallel.
// Sequential summation of n terms is off by at most n * 2^-53 * (sum of magnitudes) from the exact sum, the tree by far
// less, so the sequential result lies in an interval around the tree's; what is stored is that result rounded to
// fp32, 2^29 times coarser, through monotone operations only.  If both ends of the interval round to the same fp32
// number, it is the sequential one's.  Otherwise (about one row in 10^5) the CTA forms the sequential sum.
constexpr uint32_t kRowThreads = 128;

__device__ __forceinline__ double cta_sum(double v, double *part) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, d));
    __syncthreads();
    if ((threadIdx.x & 31u) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = part[0];
#pragma unroll
    for (uint32_t i = 1; i < kRowThreads / 32u; ++i) s = __dadd_rn(s, part[i]);
    return s;                                    // the same in every thread
}
// how far the sequential sum of n terms (magnitudes summing to `mag`) can be from the tree's
__device__ __forceinline__ double order_bound(uint32_t n, double mag) { return (1.02 * double(n) + 64.0) * kUnit * mag; }

__device__ __forceinline__ float rms_result(double acc, uint32_t C) {
    double m = __dsqrt_rn(__ddiv_rn(acc, double(C)));
    if (!(m > 1e-12)) m = 1e-12;
    return __double2float_rn(m);
}

// The first kClearCtas CTAs clear the state and the histograms of the search (as memsets before this kernel they and their gaps took 10 us).
constexpr uint32_t kClearCtas = 148;
__global__ void __launch_bounds__(kRowThreads) row_rms_kernel(const float *__restrict__ W, uint32_t C, float *__restrict__ mu, uint4 *__restrict__ clear, uint32_t n_clear) {
    __shared__ double part[kRowThreads / 32];
    __shared__ __align__(16) float4 stage[kRowThreads];
    const uint32_t tid = threadIdx.x, n4 = C / 4;
    if (blockIdx.x < kClearCtas) {
#pragma unroll 4
        for (uint32_t i = blockIdx.x * kRowThreads + tid; i < n_clear; i += kClearCtas * kRowThreads) clear[i] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    const uint32_t row = blockIdx.x - kClearCtas;
    const float4 *x = reinterpret_cast<const float4 *>(W + size_t(row) * C);   // 16-byte aligned: C % 8 == 0
    double acc = 0.0;
    auto add = [&](const float4 v) {
        const double a = double(v.x), b = double(v.y), c = double(v.z), d = double(v.w);
        acc = __fma_rn(a, a, acc);               // (squares of fp32 numbers are exact in double)
        acc = __fma_rn(b, b, acc);
        acc = __fma_rn(c, c, acc);
        acc = __fma_rn(d, d, acc);
    };
    uint32_t j = tid;
    for (; j + 3u * kRowThreads < n4; j += 4u * kRowThreads) {
        const float4 a = __ldg(x + j), b = __ldg(x + j + kRowThreads), c = __ldg(x + j + 2u * kRowThreads), d = __ldg(x + j + 3u * kRowThreads);
        add(a); add(b); add(c); add(d);
    }
    for (; j < n4; j += kRowThreads) add(__ldg(x + j));
    const double sum = cta_sum(acc, part), off = order_bound(C, sum);
    const float lo = rms_result(__dsub_rn(sum, off), C), hi = rms_result(__dadd_rn(sum, off), C);
    if (lo == hi) {
        if (tid == 0) mu[row] = lo;
        return;
    }
    acc = 0.0;                                   // index order
    for (uint32_t j0 = 0; j0 < n4; j0 += kRowThreads) {
        __syncthreads();
        if (j0 + tid < n4) stage[tid] = __ldg(x + j0 + tid);
        __syncthreads();
        if (tid == 0)
            for (uint32_t i = 0, n = min(kRowThreads, n4 - j0); i < n; ++i) {
                const float4 v = stage[i];
                acc = __dadd_rn(acc, __dmul_rn(double(v.x), double(v.x)));
                acc = __dadd_rn(acc, __dmul_rn(double(v.y), double(v.y)));
                acc = __dadd_rn(acc, __dmul_rn(double(v.z), double(v.z)));
                acc = __dadd_rn(acc, __dmul_rn(double(v.w), double(v.w)));
            }
    }
    if (tid == 0) mu[row] = rms_result(acc, C);
}

// ---- E8 quantisation (Eq. 2-4) ---------------------------------------------------------------------------
// Eq. 3 on one 8-vector: integer point and fp32 residuals of that point
struct D8 {
    int32_t z[8];
    float res[8];
};
__device__ __forceinline__ void nearest_d8(const float *y, D8 &o) {
    int32_t sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float f = rintf(y[i]);                 // ties to even
        o.z[i] = int32_t(f);
        o.res[i] = __fsub_rn(y[i], f);
        sum += o.z[i];
    }
    if (sum & 1) {
        int at = 0;
        float big = fabsf(o.res[0]);
#pragma unroll
        for (int i = 1; i < 8; ++i) {
            const float a = fabsf(o.res[i]);
            if (a > big) { big = a; at = i; }        // first coordinate of largest residual
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i == at) {
                o.z[i] += (o.res[i] >= 0.0f) ? 1 : -1;   // sign(0) = +1
                o.res[i] = __fsub_rn(y[i], float(o.z[i]));
            }
    }
}

// Eq. 2 as the host writes it: z[0..8) = the lattice point's integer parts, returns the coset; -1 if a coordinate leaves
// the histogram range
__device__ __noinline__ int quantise_exact(const float *x, float mu, float s, int32_t *z) {
    float y[8], yh[8];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        y[i] = __fdiv_rn(__fdiv_rn(x[i], mu), s);
        yh[i] = __fsub_rn(y[i], 0.5f);
        ok = ok && (fabsf(y[i]) < 4000.0f);
    }
    if (!ok) return -1;
    D8 a, h;
    nearest_d8(y, a);
    nearest_d8(yh, h);
    double da = 0.0, dh = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        da = __dadd_rn(da, __dmul_rn(double(a.res[i]), double(a.res[i])));
        dh = __dadd_rn(dh, __dmul_rn(double(h.res[i]), double(h.res[i])));
    }
    const bool half = dh < da;                       // the half coset only when strictly closer
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = half ? h.z[i] : a.z[i];
    return half ? 1 : 0;
}

// two fp32 numbers per instruction
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
// a - b, exactly fp32's: b's sign flips without rounding
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tsub.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float rcp_approx(float v) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(v));            // within 2^-23
    return r;
}
// The same point from y ~ x * r with r ~ 1 / (mu s), or `false` where the difference could matter.  z comes back as the
// bits of 1.5 * 2^23 + z.
// y is within E = 5e-7 (|y| + 1) of the host's (two roundings of 2^-24 there; a product, a reciprocal within 2^-23
// and a product here; and y - 1/2 on either side).
// With a_i = |y_i - rint(y_i)|: the integer candidate has residuals a_i, the half candidate 1/2 - a_i, and Eq. 3's parity
// step moves the largest residual r to 1 - r; so the squared distances differ by
//     d_half - d_int = 2 - sum a + [half parity odd] 2 min a - [integer parity odd] (1 - 2 max a).
// Every decision - the two roundings of each coordinate, the coset, which coordinate the parity step moves - must have
// a margin of more than what E can change.  At 4 bpp one block in 3000 fails and takes the divisions; at 8 bpp one
// in 200.  (Compared with the exact routine on 6 x 10^7 random blocks and blocks built around ties: no difference.)
// About 17 instructions per coordinate, most on the multiply-add pipe, two coordinates at a time where possible.
__device__ __forceinline__ bool quantise_fast(const float (&x)[8], float r, uint32_t (&z)[8], uint32_t &half) {
    const float2 magic = make_float2(12582912.0f, 12582912.0f), rr = make_float2(r, r);   // 1.5 * 2^23: rounds to the nearest integer
    float2 y[4];
    uint32_t parity = 0, signs = 0;
    float ymax = 0.0f, big = 0.0f, small = 1.0f, sum = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        y[i] = mul2(make_float2(x[2 * i], x[2 * i + 1]), rr);
        const float2 t = add2(y[i], magic), res = sub2(y[i], sub2(t, magic));
        parity ^= __float_as_uint(t.x) ^ __float_as_uint(t.y);
        signs ^= __float_as_uint(res.x) ^ __float_as_uint(res.y);
        ymax = fmaxf(fmaxf(ymax, fabsf(y[i].x)), fabsf(y[i].y));
        big = fmaxf(fmaxf(big, fabsf(res.x)), fabsf(res.y));
        small = fminf(fminf(small, fabsf(res.x)), fabsf(res.y));
        sum += fabsf(res.x) + fabsf(res.y);
    }
    const bool odd_int = parity & 1u, odd_half = (parity ^ (signs >> 31)) & 1u;
    const float E = 5e-7f * ymax + 5e-7f;
    float d = 2.0f - sum;
    if (odd_half) d += 2.0f * small;
    if (odd_int) d -= 1.0f - 2.0f * big;
    const bool h = d < 0.0f, odd = h ? odd_half : odd_int;
    half = h ? 1u : 0u;
    const bool ok = small > E && big < 0.5f - E && fabsf(d) > 16.0f * E + 4e-6f && ymax < 3990.0f;
    // the chosen candidate: y or y - 1/2 rounded, its largest residual moved away from y if the coordinate sum is odd
    const float shift = h ? -0.5f : 0.0f;
    const float most = odd ? (h ? 0.5f - small : big) - 2.5f * E : 2.0f;
    float hits = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 v = add2(y[i], make_float2(shift, shift));
        float2 t = add2(v, magic);
        const float2 res = sub2(v, sub2(t, magic));
        if (fabsf(res.x) >= most) { hits += 1.0f; t.x += __uint_as_float((__float_as_uint(res.x) & 0x80000000u) | 0x3F800000u); }
        if (fabsf(res.y) >= most) { hits += 1.0f; t.y += __uint_as_float((__float_as_uint(res.y) & 0x80000000u) | 0x3F800000u); }
        z[2 * i] = __float_as_uint(t.x);
        z[2 * i + 1] = __float_as_uint(t.y);
    }
    return ok && !(odd && hits != 1.0f);
}

// ---- counting passes ---------------------------------------------------------------------------------------
// A pass quantises the listed rows (all rows) at a scale and counts the fields.  The whole search of Algorithm 1 and
// the rate correction after it are one stream of launches with one wait at the end: the last CTA of a pass evaluates
// Eq. 10-12 on the counts and leaves the next scale in device memory.
//
// A pass costs about 12 us whatever the sample (launch, clearing and flushing counters, the evaluation's chain of dependent reads), and
// counting 2^18 blocks of a sample only 4 us more.  So a pass counts and evaluates several scales at once, each by CTAs of its own, and the
// last CTA to finish takes as many steps of the bisection as it has scales for.  Which scales a step looks at depends on the
// steps before it, but where they lead can be foretold: after the first step by the one-bit-per-doubling law of Eq. 9, later by
// interpolation between the ends of the bracket.  The scales of a pass are those that the bisection meets if the target is at the foretold
// scale, or a little to either side of it; a step whose scale is not among them is left to the next pass.  No decision depends on
// the forecast.  Where the passes that are left could not end the bisection one step at a time, a pass takes the whole tree of its next
// four steps, fifteen scales; that many passes are launched that this always ends it, and those that find it ended cost 2 us each.
// Twelve steps usually take three passes.  (Fixed trees: 1, 2, 3, 3, 3 steps per launch, for samples up to 2^17 blocks 1, 3, 4, 4.  The
// first launches took fewer steps because the outer scales of a wide bracket are so fine - s = 0.003 - that all they count goes to
// global memory, 120 us for 2^18 blocks; the forecast does not look at them.)
//
// Counting: nine increments per block, most of them of a few values around zero.  Each lane has its own column of
// counters for those (bank = lane: no two lanes of a warp meet), values up to +-256 go to a plain window, the rest to
// global memory.
constexpr uint32_t kCountThreads = 1024;
constexpr int kHotBins = 32, kHotOrigin = -16;   // values with a counter column per lane, per coordinate table
constexpr uint32_t kHotStride = (kHotBins + 1) * 32;   // words per table: one more row takes what lies outside
constexpr int kWinBins = 512, kWinOrigin = -256; // values with one counter per CTA, per table (2048 of them gain nothing at 8 bpp either)
constexpr uint32_t kHotWords = 16 * kHotStride, kWinWords = EP_NUM_TABLES * kWinBins;
// Symbols over all tables that an evaluation holds in shared memory (it reuses the counters' space; 196 KB for 49152 of them
// cost the passes 4 % of their time).  A scale of the search with more - heavy tails meet some at 6 bpp - is judged by the
// entropy of its counts if that is enough, as it is for scales that are far too fine; if not the host takes over.
constexpr uint32_t kEvalSymbols = kHotWords + kWinWords;
constexpr uint32_t kManySymbols = 8192;          // with more the counts' entropy is looked at first (see gather_counts)
constexpr uint32_t kCountSmem = 4 * kEvalSymbols;
constexpr uint32_t kFirstCounts = 6144;          // counts that come back with the state; more take a second copy
constexpr uint32_t kLevels = 4, kCandidates = (1u << kLevels) - 1u;   // a whole tree of steps

// Symbols' entries by (coset, field, value): the two cosets' tables of a field have the same range here (the wider of
// both ends), so that the second coset's entries follow at one distance.
struct EncodeTables {
    uint32_t base[9];                // byte offset of value 0's entry of field k (0: the coset) under coset 0, modulo 2^32
    uint32_t coset;                  // bytes from coset 0's entries to coset 1's
    uint32_t total;                  // entries
};

// What Eq. 17 needs of a symbol, without a division: x / f for x < 2^31 is umulhi(x, rcp) >> sh with
// sh = ceil(log2 f) - 1 and rcp = ceil(2^(32 + sh) / f) (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994; exact for 31-bit x).  f = 1 takes rcp = 2^32 - 1, which gives x - 1, and an offset that
// makes up for it.  With q = x / f the new state is q 2^b + x mod f + F = x + (2^b - f) q + F.
// {rcp, first state that gives off a word: f 2^(31-b), 2^b - f, sh | offset << 16}
__device__ __forceinline__ uint4 encode_entry(uint32_t fF, uint32_t b) {
    const uint32_t M = 1u << b, f = max(fF & 0xFFFFu, 1u), F = fF >> 16;
    if (f == 1u) return make_uint4(0xFFFFFFFFu, 1u << (31u - b), M - 1u, (F + M - 1u) << 16);
    const uint32_t sh = 31u - __clz(int(f - 1u));
    // (the quotient has at most 32 integer bits and a fraction of at least 1 / f: its ceiling is right in double)
    const uint32_t rcp = uint32_t(ceil(__ddiv_rn(double(1ull << (32u + sh)), double(f))));
    return make_uint4(rcp, f << (31u - b), M - f, sh | (F << 16));
}

struct CountDir { int32_t lo[EP_NUM_TABLES]; uint32_t K[EP_NUM_TABLES]; };

// one scale of a pass (device memory)
struct Candidate {
    CountDir dir;
    // observed range, stored as the larger of (kHistBins - bin) and of (bin + 1); 0: none
    uint32_t from[EP_NUM_TABLES], to[EP_NUM_TABLES];
    uint32_t finished;               // its CTAs that are done
    uint32_t overflow;               // a coordinate left the histogram range
};
// A candidate's verdict, four bits: a b-bit table exists; the rate lies above the target; too close to say (with kAbove, without kValid: a table
// exists, but the counts were not kept); a coordinate left the histogram range.  A pass's verdicts come together in one 64-bit word: the
// candidates' last CTAs add theirs and a one to its highest four bits, so that the one whose addition was the last has them all in hand.
constexpr uint32_t kValid = 1, kAbove = 2, kUndecided = 4, kOverflow = 8, kNoCounts = kAbove | kUndecided;
static_assert(kCandidates == kMostScales, "fifteen verdicts and their count in 64 bits");
// what the passes leave for one another and for the host (device memory, zeroed before a search)
struct SearchState {
    double lo, hi;                   // the bracket,
    double rate_lo, rate_hi;         // the rates at its ends (NaN: not known)
    double mid[kCandidates], rate[kCandidates];   // scales of the next or running pass, and their rates
    uint32_t scales, left;           // how many scales, with the pass that counts them (scales_word; 0: the bisection has ended), steps still to take
    double last_log_s, last_rate;    // rate correction: the last point
    unsigned long long verdicts;     // of the running pass's candidates
    float s;                         // the next pass's scale
    float s_counted;                 // the scale of the full counts
    uint32_t has_last, lost;         // a step's rate was evaluated; `last` does not hold the counts of the last such step
    uint32_t undecided;              // a decision within the rounding error, or too many symbols: the host repeats the search
    uint32_t overflow;               // a coordinate left the histogram range
    uint32_t stop;                   // the full passes are over
    uint32_t polished;               // ... because the rate correction ended (0: the tensor overflows the tables, the host decides)
    CountDir last, full;
    EncodeTables coder;              // tile coding: where the symbols' entries are,
    uint32_t code;                   //              whether they are there and the tiles are to be coded,
    uint32_t tiles_done;             //              CTAs of the launch that are done
    uint32_t reported;               // CTAs that have brought their share of this and of the counts to the host
    Candidate cand[kCandidates];
};
constexpr size_t kStateBytes = 8192;
static_assert(sizeof(SearchState) <= kStateBytes, "state area");

// the constants of Eq. 10-12
struct RateParams {
    double target, retained_bits_total, fixed_bits, weights, fields;   // fixed_bits: restarts, scales, header
    int32_t b;
};
enum PassMode { kPassCount, kPassSearch, kPassPolish };   // counts only; steps of the bisection; a pass of the rate correction

struct CountParams {
    const float *W;
    const float *mu;
    const uint32_t *rows;            // null: all rows
    uint4 *fields;                   // one per block: z1 .. z7 and 2 m + c as int16; null: not kept
    uint32_t *hist;                  // per candidate EP_NUM_TABLES x kHistBins, zero between passes
    SearchState *state;
    uint32_t *cand_counts;           // per candidate kEvalSymbols
    uint32_t *last_counts, *full_counts;
    uint4 *entries;                  // rate correction: the tile coder's entries, made by the pass that ends it, and
    uint32_t *full_freq;             // the frequencies they are of (null: not wanted)
    uint32_t n_blocks, C, per_row;
    uint32_t mode;
    uint32_t pass;                   // of the search; the first, 0, counts one scale, the middle of the bracket {lo0, hi0}
    uint32_t steps;                  // first pass of the search: steps to take
    uint32_t most;                   // scales of the next pass, at most, and
    uint32_t after;                  // passes of the search behind the next one
    float s;                         // mode kPassCount
    RateParams rate;
    double lo0, hi0;                 // the search bracket
    int32_t step, last_step;         // rate correction: passes done so far, and allowed
};

__device__ __forceinline__ uint32_t warp_sum(uint32_t v) { return __reduce_add_sync(0xFFFFFFFFu, v); }
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, d));
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    return v;
}

// bracket of candidate k: the tree's nodes in heap order, the left child of a node being the outcome "rate above target"
__device__ __forceinline__ void bracket_of(uint32_t k, double &lo, double &hi) {
    const uint32_t n = k + 1u;
    for (int bit = 30 - __clz(int(n)); bit >= 0; --bit) {
        const double mid = __dsqrt_rn(__dmul_rn(lo, hi));
        if ((n >> bit) & 1u) hi = mid; else lo = mid;
    }
}

// Eq. 10-11 for a given C_CE, as the host computes it (everything but the first difference is exact)
__device__ __forceinline__ double bits_at(const RateParams &P, double tables, double cce) {
    const double left = fmax(0.0, __dsub_rn(cce, P.retained_bits_total));
    return __dadd_rn(__dadd_rn(__dmul_rn(16.0, ceil(__dmul_rn(left, 0.0625))), P.fixed_bits), tables);
}

// C_CE below is a sum in another order, with this device's log2 (within one unit in the last place; terms of at most 15 bits
// per field, a few thousand additions).  How far the host's can be:
__device__ __forceinline__ double cce_bound(const RateParams &P, double cce) { return 1e-11 * (cce + 16.0 * P.fields); }

struct Evaluation { double cce, tables; uint32_t worst; bool too_many, above; };   // above: by the counts' entropy alone

struct Ranges { int32_t lo[EP_NUM_TABLES]; uint32_t K[EP_NUM_TABLES], at[EP_NUM_TABLES + 1]; };    // a candidate's tables and where they start

// All threads of a candidate's last CTA: ranges and offsets of its tables, counts to `out`, histogram back to zero; unless
// only counts are wanted, the frequencies of Sec. 3.3 (integers: the host's exactly), C_CE of Eq. 8 and the largest alphabet.
__device__ __forceinline__ Evaluation gather_counts(const CountParams &P, uint32_t k, uint32_t *out, uint32_t *f_of, Ranges &D) {
    int32_t *const lo_of = D.lo;
    uint32_t *const K_of = D.K, *const at_of = D.at;
    __shared__ uint32_t seen_of[EP_NUM_TABLES];
    __shared__ double bits_of[EP_NUM_TABLES];
    Candidate &S = P.state->cand[k];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    if (warp == 0) {
        uint32_t K = 0;
        int32_t lo = 0;
        if (lane < EP_NUM_TABLES) {
            const uint32_t a = __ldcg(&S.from[lane]), z = __ldcg(&S.to[lane]);
            const uint32_t first = kHistBins - a;
            lo = a ? kHistOrigin + int32_t(first) : 0;
            K = a ? z - first : 0u;                         // z = last bin + 1
            S.from[lane] = 0;
            S.to[lane] = 0;
            S.dir.lo[lane] = lo;
            S.dir.K[lane] = K;
        }
        uint32_t incl = K;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= uint32_t(d)) incl += n;
        }
        if (lane < EP_NUM_TABLES) { lo_of[lane] = lo; K_of[lane] = K; at_of[lane + 1] = incl; }
        if (lane == 0) { at_of[0] = 0; S.finished = 0; }
    }
    __syncthreads();
    const bool evaluate = P.mode != kPassCount;
    Evaluation E;
    // a scale of the search with this many symbols is usually far too fine: the entropy of its counts says so for less
    const bool many = P.mode == kPassSearch && at_of[EP_NUM_TABLES] > kManySymbols;
    double total = 0.0;
    E.cce = 0.0;
    E.worst = 0;
    E.above = false;
    E.too_many = at_of[EP_NUM_TABLES] > kEvalSymbols;       // (only full_counts has room for more)
    E.tables = 8.0 * double((8u * EP_NUM_TABLES + 2u * at_of[EP_NUM_TABLES] + 3u) & ~3u);
    const bool keep = !E.too_many || P.mode != kPassSearch;
    for (uint32_t t = warp; t < EP_NUM_TABLES; t += kCountThreads / 32u) {
        const uint32_t K = K_of[t], at = at_of[t];
        uint32_t *h = P.hist + (k * EP_NUM_TABLES + t) * kHistBins + (lo_of[t] - kHistOrigin);
        unsigned long long sum = 0;
        uint32_t seen = 0;
        double nlogn = 0.0;
        if (many) {
#pragma unroll 8
            for (uint32_t j = lane; j < K; j += 32) {
                const float n = float(__ldcg(h + j));
                if (n > 1.0f) nlogn += double(n) * double(log2f(n));
            }
        }
        for (uint32_t j0 = lane; j0 < K; j0 += 8u * 32u) {     // eight loads under way at a time
            uint32_t n[8];
#pragma unroll
            for (uint32_t u = 0; u < 8; ++u) n[u] = j0 + 32u * u < K ? __ldcg(h + j0 + 32u * u) : 0u;
#pragma unroll
            for (uint32_t u = 0; u < 8; ++u) {
                const uint32_t j = j0 + 32u * u;
                if (j >= K) break;
                h[j] = 0;
                if (keep) out[at + j] = n[u];
                if (!E.too_many) f_of[at + j] = n[u];
                sum += n[u];
                seen += n[u] != 0;
            }
        }
        if (!evaluate) continue;
        total = double(warp_sum(sum));
        seen = warp_sum(seen);
        if (many) nlogn = warp_sum(nlogn);
        if (lane == 0) { bits_of[t] = many && total > 0.0 ? total * log2(total) - nlogn : 0.0; seen_of[t] = seen; }
    }
    if (many) {
        __syncthreads();
        double least = -1e-5 * P.rate.fields;                // log2f: an error of 2e-6 per count
        for (uint32_t t = 0; t < EP_NUM_TABLES; ++t) { least += bits_of[t]; E.worst = max(E.worst, seen_of[t]); }
        E.above = __ddiv_rn(bits_at(P.rate, E.tables, least - cce_bound(P.rate, least)), P.rate.weights) > P.rate.target;
        if (E.above || E.too_many) return E;
        __syncthreads();
    }
    if (evaluate && !E.too_many && warp < EP_NUM_TABLES) {
        const uint32_t t = warp, K = K_of[t], at = at_of[t];
        // frequencies: max(1, floor(n 2^b / total)), then the deficit to the largest or the excess from the largest
        const uint32_t M = 1u << P.rate.b;
        uint32_t fsum = 0, best = 0;
        auto key = [](uint32_t f, uint32_t j) { return (f << 16) | (0xFFFFu - j); };      // f <= 2^15, j < 2^13: first of the largest
        // (one division per table instead of one per symbol, and four symbols' chains side by side: the passes of 10240 x 3840
        // at 4 bpp, first to last, 258.1 -> 254.8 us, of 480 x 7512 at 8 bpp 333.2 -> 327.4)
        const double per_total = __ddiv_rn(1.0, total);      // (not used for an empty table)
#pragma unroll 4
        for (uint32_t j = lane; j < K; j += 32) {
            const uint32_t n = f_of[at + j];
            uint32_t f = 0;
            if (n) {
                const double nM = double(n) * double(M);                                  // below 2^47: exact
                uint32_t q = uint32_t(nM * per_total);                                    // off by one at most: 2^15 times 2^-52
                const double r = __fma_rn(-double(q), total, nM);                         // exact
                if (r < 0.0) --q; else if (r >= total) ++q;
                f = max(q, 1u);
            }
            f_of[at + j] = f;
            fsum += f;
            best = max(best, key(f, j));
        }
        fsum = warp_sum(fsum);
        best = __reduce_max_sync(0xFFFFFFFFu, best);
        __syncwarp();
        if (K && fsum < M) {
            if (lane == 0) f_of[at + 0xFFFFu - (best & 0xFFFFu)] += M - fsum;
        }
        // A turn takes as much as it can from the first of the largest.  An alphabet of thousands with a count of one each, all
        // raised to a frequency of one, needs hundreds of turns: after two the rest is taken in the same order at once.
        for (uint32_t turn = 0; K && fsum > M; ++turn) {
            const uint32_t f = best >> 16, excess = fsum - M, take = min(excess, f - 1u);
            if (f <= 1u) break;                              // more symbols than slots: judged by `worst`
            if (turn == 2u) {
                // the smallest `top` for which the frequencies above it, all lowered to one, give no more than the excess
                uint32_t low = 1u, top = f, taken = 0;
                while (low < top) {
                    const uint32_t mid = (low + top) >> 1;
                    uint32_t more = 0;
#pragma unroll 8
                    for (uint32_t j = lane; j < K; j += 32) more += f_of[at + j] > mid ? f_of[at + j] - 1u : 0u;
                    more = warp_sum(more);
                    if (more <= excess) { top = mid; taken = more; } else low = mid + 1u;
                }
                // of those that equal it the first ones give the rest
                uint32_t before = 0;
                for (uint32_t j0 = 0; j0 < K; j0 += 32) {
                    const uint32_t j = j0 + lane, g = j < K ? f_of[at + j] : 0u;
                    const bool equal = g == top && top > 1u;
                    const uint32_t same = __ballot_sync(0xFFFFFFFFu, equal);
                    const uint32_t gone = taken + (before + __popc(same & ((1u << lane) - 1u))) * (top - 1u);
                    if (g > top) f_of[at + j] = 1u;
                    else if (equal && gone < excess) f_of[at + j] = top - min(excess - gone, top - 1u);
                    before += __popc(same);
                }
                break;
            }
            if (lane == 0) f_of[at + 0xFFFFu - (best & 0xFFFFu)] = f - take;
            fsum -= take;
            __syncwarp();
            if (fsum <= M) break;
            best = 0;
#pragma unroll 4
            for (uint32_t j = lane; j < K; j += 32) best = max(best, key(f_of[at + j], j));
            best = __reduce_max_sync(0xFFFFFFFFu, best);
        }
        __syncwarp();
        double bits = 0.0;
#pragma unroll 4
        for (uint32_t j = lane; j < K; j += 32) {
            const uint32_t f = f_of[at + j];
            if (f) bits += double(out[at + j]) * (double(P.rate.b) - log2(double(f)));
        }
        bits = warp_sum(bits);
        if (lane == 0) bits_of[t] = bits;
    }
    __syncthreads();
    if (evaluate && warp == 0) {
        E.cce = warp_sum(lane < EP_NUM_TABLES ? bits_of[lane] : 0.0);
        E.worst = __reduce_max_sync(0xFFFFFFFFu, lane < EP_NUM_TABLES ? seen_of[lane] : 0u);
    }
    return E;                                                // (cce and worst in warp 0)
}
// warp 0 after a candidate of the search is gathered: is its rate above the target?  The verdict in lane 0, the rate in lane 1
__device__ __forceinline__ uint32_t judge_candidate(const CountParams &P, uint32_t k, const Evaluation &E, double &rate) {
    // lane 1 at the estimate, lanes 0 and 2 at the ends of its interval
    const uint32_t lane = threadIdx.x & 31u, overflow = __ldcg(&P.state->cand[k].overflow);
    const double cce = E.cce + (double(lane) - 1.0) * cce_bound(P.rate, E.cce);
    rate = __ddiv_rn(bits_at(P.rate, E.tables, cce), P.rate.weights);
    const uint32_t b = __ballot_sync(0xFFFFFFFFu, rate > P.rate.target) & 7u;
    uint32_t v = kValid | ((b & 2u) ? kAbove : 0u) | ((b == 0u || b == 7u) ? 0u : kUndecided);
    if (E.above) v = E.too_many ? kNoCounts : kAbove | kValid;
    else if (E.too_many) v = kUndecided;
    if (E.worst > (1u << P.rate.b)) v = kAbove;                  // no b-bit table exists for this scale: too fine
    if (E.above || E.too_many || v == kAbove) rate = nan("");    // not known
    return v | (overflow ? kOverflow : 0u);
}

// Warp 0 of a pass's last CTA: as many steps as the pass's n scales are for, in order, and the scales of the next pass.  Returns (in every lane) the
// candidate whose counts are to be kept, or -1: the host gets those of the last step whose scale had a table.  That step is usually one of the
// last pass, but while the bracket's finer end has no table, all steps of the next pass may be without one.  (Kept by the last pass only, 4 of 24 searches
// at 9 bits - 96 x 1024, Laplace, for a rate above that of the finest scale with a table - were left to the host, 9 of 24 with Student-t rows.)
__device__ __noinline__ int32_t take_steps(const CountParams &P, uint32_t n, unsigned long long verdicts) {
    SearchState &S = *P.state;
    const bool first_pass = P.pass == 0u;
    const uint32_t lane = threadIdx.x & 31u;
    const double nothing = nan("");
    double lo = first_pass ? P.lo0 : __ldcg(&S.lo), hi = first_pass ? P.hi0 : __ldcg(&S.hi);
    double rate_lo = first_pass ? nothing : __ldcg(&S.rate_lo), rate_hi = first_pass ? nothing : __ldcg(&S.rate_hi);
    uint32_t left = first_pass ? P.steps : __ldcg(&S.left), undecided = 0, overflow = 0;
    // lane k: scale, verdict and rate of candidate k
    const double scale = lane >= n ? -1.0 : first_pass ? __dsqrt_rn(__dmul_rn(lo, hi)) : __ldcg(&S.mid[min(lane, kCandidates - 1u)]);
    const double rate = __ldcg(&S.rate[min(lane, kCandidates - 1u)]);
    const uint32_t verdict = uint32_t(verdicts >> (4u * min(lane, kCandidates - 1u))) & 15u;
    int32_t last = -1;
    while (left) {
        const double mid = __dsqrt_rn(__dmul_rn(lo, hi));
        const uint32_t at = __ballot_sync(0xFFFFFFFFu, scale == mid);
        if (!at) break;
        const uint32_t k = uint32_t(__ffs(int(at)) - 1), v = __shfl_sync(0xFFFFFFFFu, verdict, int(k)), kind = v & (kValid | kAbove | kUndecided);
        const double r = __shfl_sync(0xFFFFFFFFu, rate, int(k));
        overflow |= v & kOverflow;
        undecided |= kind != kNoCounts && (v & kUndecided);
        if (v & kValid) last = int32_t(k);
        if (kind == kNoCounts) last = -2;
        if (v & kAbove) { lo = mid; rate_lo = r; } else { hi = mid; rate_hi = r; }
        --left;
    }
    const bool keep = last >= 0 && (!left || rate_lo != rate_lo);
    const uint32_t lost = last == -1 ? (first_pass ? 0u : __ldcg(&S.lost)) : !keep;
    if (lane == 0) {
        S.lo = lo;
        S.hi = hi;
        S.rate_lo = rate_lo;
        S.rate_hi = rate_hi;
        S.left = left;
        S.s = __double2float_rn(__dsqrt_rn(__dmul_rn(lo, hi)));
        S.verdicts = 0;
        if (overflow) S.overflow = 1;
        if (undecided) S.undecided = 1;
        if (last != -1) S.has_last = 1;
        S.lost = lost;
        if (!left && lost) S.undecided = 1;
    }
    if (!left) {
        if (lane == 0) S.scales = scales_word(P.pass + 1u, 0u);
        return keep ? last : -1;
    }
    // the next pass's scales.  The forecast is in fp32 (in double it took 7 us); the scales themselves are the bisection's, to the bit
    uint32_t next = 0;
    const float x_lo = log2f(float(lo)), x_hi = log2f(float(hi)), width = x_hi - x_lo, target = float(P.rate.target), r_lo = float(rate_lo), r_hi = float(rate_hi);
    const bool both = r_lo > r_hi;
    // (the rate bends by a few hundredths of a bit per doubling of the scale and doubling)
    const float off = both ? fmaxf(0.004f, 0.04f * width * width) : 0.12f;
    const float x = both ? x_lo + width * __fdividef(r_lo - target, r_lo - r_hi) : r_lo == r_lo ? x_lo + (r_lo - target) : x_hi - (target - r_hi);
    if (x == x && left - 1u <= kLevels * P.after) {
        // lanes 0, 1, 2 follow the bisection to the foretold scale and to either side of it
        __shared__ double path[30];
        const float to = exp2f(x + (lane == 1u ? off : lane == 2u ? -off : 0.0f));
        double a = lo, b = hi;
        float w = width;
        uint32_t levels = 0;
        for (; levels < min(left, 10u) && w > 0.5f * off; ++levels, w *= 0.5f) {
            const double mid = __dsqrt_rn(__dmul_rn(a, b));
            if (lane < 3u) path[3u * levels + lane] = mid;
            if (float(mid) < to) a = mid; else b = mid;
        }
        __syncwarp();
        // step by step, the two others where they differ from the first
        const double mine = lane < 3u * levels ? path[lane] : 0.0, first = lane < 3u * levels ? path[lane - lane % 3u] : 0.0;
        const bool want = lane < 3u * levels && (lane % 3u == 0u || mine != first);
        const uint32_t wanted = __ballot_sync(0xFFFFFFFFu, want), at = __popc(wanted & ((1u << lane) - 1u));
        if (want && at < P.most) S.mid[at] = mine;
        next = min(uint32_t(__popc(wanted)), P.most);
    }
    if (!next) {
        next = (1u << min(left, kLevels)) - 1u;
        double a = lo, b = hi;
        bracket_of(min(lane, kCandidates - 1u), a, b);
        if (lane < next) S.mid[lane] = __dsqrt_rn(__dmul_rn(a, b));
    }
    if (lane == 0) S.scales = scales_word(P.pass + 1u, next);
    return keep ? last : -1;
}
// All threads: the host reports the rate of the last evaluated step - its counts, until a later one's replace them
__device__ __forceinline__ void keep_last(const CountParams &P, uint32_t k) {
    SearchState &S = *P.state;
    const Candidate &c = S.cand[k];
    uint32_t n = 0;
    for (int t = 0; t < EP_NUM_TABLES; ++t) n += __ldcg(&c.dir.K[t]);
    for (uint32_t i = threadIdx.x; i < n; i += kCountThreads) P.last_counts[i] = __ldcg(P.cand_counts + size_t(k) * kEvalSymbols + i);
    if (threadIdx.x < EP_NUM_TABLES) {
        S.last.lo[threadIdx.x] = __ldcg(&c.dir.lo[threadIdx.x]);
        S.last.K[threadIdx.x] = __ldcg(&c.dir.K[threadIdx.x]);
    }
}

// thread 0 after a full pass: the rate correction's next scale, or its end (run_encode has the same steps)
__device__ void polish(const CountParams &P, float s, const Evaluation &E) {
    SearchState &S = *P.state;
    S.s_counted = s;
    if (E.worst > (1u << P.rate.b)) {                            // before the first move: the host raises b or s
        if (P.step > 0) S.undecided = 1;
        S.stop = 1;
        return;
    }
    if (E.too_many) { S.undecided = 1; S.stop = 1; return; }
    S.polished = 1;
    if (P.step >= P.last_step) { S.stop = 1; return; }
    const double off = cce_bound(P.rate, E.cce), bits = bits_at(P.rate, E.tables, E.cce);
    // the payload estimate is rounded up to words: if it is the same at both ends of the interval it is the host's exactly
    if (bits_at(P.rate, E.tables, E.cce - off) != bits_at(P.rate, E.tables, E.cce + off)) { S.undecided = 1; S.stop = 1; return; }
    const double est = __ddiv_rn(bits, P.rate.weights);
    if (fabs(__dsub_rn(est, P.rate.target)) <= __dmul_rn(0.002, P.rate.target)) { S.stop = 1; return; }
    const double log_s = log2(double(s));
    double per_doubling = 1.0;
    if (P.step > 0 && log_s != S.last_log_s) {
        per_doubling = -__ddiv_rn(__dsub_rn(est, S.last_rate), __dsub_rn(log_s, S.last_log_s));
        if (!(per_doubling >= 0.5)) per_doubling = 0.5;
        if (per_doubling > 4.0) per_doubling = 4.0;
    }
    // log2 and exp2 may differ from the host's in the last place; 1e-10 is far above what that makes of an ordinary move
    const double near = fmax(1e-10, next_scale_error(log_s, S.last_log_s, P.step > 0, __dsub_rn(est, P.rate.target), per_doubling));
    S.last_log_s = log_s;
    S.last_rate = est;
    const double moved = exp2(__dadd_rn(log_s, __ddiv_rn(__dsub_rn(est, P.rate.target), per_doubling)));
    auto next = [&](double m) {
        if (!(m >= P.lo0)) m = P.lo0;
        if (m > P.hi0) m = P.hi0;
        return __double2float_rn(m);
    };
    const float to = next(moved);
    if (next(moved * (1.0 - near)) != to || next(moved * (1.0 + near)) != to) { S.undecided = 1; S.stop = 1; return; }
    if (to == s) { S.stop = 1; return; }
    S.s = to;
}

// All threads of the CTA that ended the rate correction: the tile coder's entries of the frequencies that gather_counts left in
// shared memory, laid out as coder_layout does, so that coding starts without the host's tables (which are the same numbers: the
// host compares them).  Alphabets beyond the coder's shared memory are left to the host.
__device__ __noinline__ void make_coder(const CountParams &P, const uint32_t *f_of, const Ranges &D) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    int32_t lo = 0, hi = 0;                      // lane k: field k
    if (lane >= 1u && lane < 9u) {
        bool any = false;
#pragma unroll
        for (uint32_t c = 0; c < 2u; ++c) {
            const uint32_t t = 8u * c + lane;
            if (!D.K[t]) continue;
            const int32_t end = D.lo[t] + int32_t(D.K[t]);
            lo = any ? min(lo, D.lo[t]) : D.lo[t];
            hi = any ? max(hi, end) : end;
            any = true;
        }
    }
    uint32_t upto = uint32_t(hi - lo);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, upto, d);
        if (lane >= uint32_t(d)) upto += n;
    }
    const uint32_t first = upto - uint32_t(hi - lo), size = __shfl_sync(0xFFFFFFFFu, upto, 31);
    if (D.at[EP_NUM_TABLES] > kMaxTableSymbols || 2u * size + 2u > kSmemEntries) return;
    if (warp < EP_NUM_TABLES) {
        const uint32_t t = warp, k = t ? ((t - 1u) & 7u) + 1u : 0u, K = D.K[t], at = D.at[t];
        const uint32_t begin = t ? (t > 8u ? size : 0u) + __shfl_sync(0xFFFFFFFFu, first, int(k)) + uint32_t(D.lo[t] - __shfl_sync(0xFFFFFFFFu, lo, int(k)))
                                 : 2u * size + uint32_t(D.lo[0]);
        uint32_t F = 0;
        for (uint32_t j0 = 0; j0 < K; j0 += 32u) {
            const uint32_t j = j0 + lane, f = j < K ? f_of[at + j] : 0u;
            uint32_t incl = f;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= uint32_t(d)) incl += n;
            }
            if (j < K) {
                P.entries[begin + j] = encode_entry(f | (F + incl - f) << 16, uint32_t(P.rate.b));
                P.full_freq[at + j] = f;
            }
            F += __shfl_sync(0xFFFFFFFFu, incl, 31);
        }
    } else if (warp == EP_NUM_TABLES && lane < 9u) {
        EncodeTables &T = P.state->coder;
        T.base[lane] = lane ? 16u * (first - uint32_t(lo)) : 32u * size;
        if (lane == 0) {
            T.coset = 16u * size;
            T.total = 2u * size + 2u;
            P.state->code = 1;
        }
    }
}

__global__ void __launch_bounds__(kCountThreads, 1) quantise_count_kernel(const __grid_constant__ CountParams P) {
    extern __shared__ __align__(16) uint32_t sm[];
    uint32_t *const hot = sm, *const win = sm + kHotWords;
    __shared__ uint32_t range_from[EP_NUM_TABLES], range_to[EP_NUM_TABLES], last_cta, ended;
    __shared__ float s_shared;
    __shared__ Ranges ranges;
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    // Launched before the previous pass has ended (see launch_count): only W, mu and rows, which are older than that, are
    // read before the wait, and only then may the next launch come up.  A pass with several scales learns behind the wait how many they are.
    const bool listed = P.mode == kPassSearch && P.pass > 0u;
    uint32_t k = 0, ctas = gridDim.x, part = blockIdx.x;                         // candidate, its CTAs and this one's share of the blocks
    uint32_t v = 0, v1 = 0, i = 0, col = 0;
    const uint32_t row_step = kCountThreads / P.per_row, col_step = kCountThreads % P.per_row;
    float4 lo4 = make_float4(0.f, 0.f, 0.f, 0.f), hi4 = lo4;
    float mu = 1.0f;
    auto load = [&]() {
        const uint32_t r = P.rows ? __ldg(P.rows + i) : i;
        const float4 *src = reinterpret_cast<const float4 *>(P.W + size_t(r) * P.C) + 2u * col;
        lo4 = __ldg(src);
        hi4 = __ldg(src + 1);
        mu = __ldg(P.mu + r);
    };
    auto begin = [&]() {
        v = uint32_t(uint64_t(P.n_blocks) * part / ctas) + tid;                  // (n_blocks < 2^31: see the launcher)
        v1 = uint32_t(uint64_t(P.n_blocks) * (part + 1u) / ctas);
        i = v / P.per_row;
        col = v - i * P.per_row;                                                 // rows of later blocks follow without divisions
        if (v < v1) load();
    };
    if (!listed) begin();
    for (uint32_t j = tid; j < (kHotWords + kWinWords) / 4u; j += kCountThreads) reinterpret_cast<uint4 *>(sm)[j] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < EP_NUM_TABLES) { range_from[tid] = 0; range_to[tid] = 0; }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (P.mode == kPassPolish && __ldcg(&P.state->stop)) return;                 // (the same for all CTAs: set by an earlier launch)
    const uint32_t scales = listed ? scales_of(__ldcg(&P.state->scales), P.pass) : 1u;
    if (!scales) return;
    if (listed) {
        const PassShare share = pass_share(gridDim.x, blockIdx.x, scales, P.n_blocks);
        k = share.scale;
        part = share.part;
        ctas = share.ctas;
        if (k >= scales) return;
        begin();
    }
    Candidate &S = P.state->cand[k];
    if (tid == 0) {
        if (listed) s_shared = __double2float_rn(__ldcg(&P.state->mid[k]));
        else if (P.mode == kPassSearch) s_shared = __double2float_rn(__dsqrt_rn(__dmul_rn(P.lo0, P.hi0)));
        else s_shared = P.mode == kPassPolish ? __ldcg(&P.state->s) : P.s;
    }
    __syncthreads();
    const float s = s_shared;
    uint32_t halves = 0, blocks = 0;
    auto count_far = [&](uint32_t t, int32_t value) {          // outside the columns
        const uint32_t w = uint32_t(value - kWinOrigin), g = uint32_t(value - kHistOrigin);
        if (w < uint32_t(kWinBins)) {
            atomicAdd(&win[t * kWinBins + w], 1u);
        } else if (g < uint32_t(kHistBins)) {
            atomicAdd(P.hist + (k * EP_NUM_TABLES + t) * kHistBins + g, 1u);
            atomicMax(&range_from[t], kHistBins - g);
            atomicMax(&range_to[t], g + 1u);
        } else {
            S.overflow = 1;
        }
    };
    while (v < v1) {
        const float x[8] = {lo4.x, lo4.y, lo4.z, lo4.w, hi4.x, hi4.y, hi4.z, hi4.w};
        const float m = mu;
        const uint32_t here = v;
        v += kCountThreads;
        i += row_step;
        col += col_step;
        if (col >= P.per_row) { col -= P.per_row; ++i; }
        if (v < v1) load();                                    // the next block is on its way while this one is worked on
        uint32_t z[8], half;                                   // coordinates as bits of 1.5 * 2^23 + z
        const float ms = __fmul_rn(m, s);
        const bool ok = quantise_fast(x, rcp_approx(ms), z, half) && ms >= 1e-30f && ms <= 1e30f;
        if (!ok) {
            float xs[8];
            int32_t zs[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) xs[j] = x[j];
            const int c = quantise_exact(xs, m, s, zs);
            if (c < 0) { S.overflow = 1; continue; }
            half = uint32_t(c);
#pragma unroll
            for (int j = 0; j < 8; ++j) z[j] = 0x4B400000u + uint32_t(zs[j]);
        }
        // Eq. 4: m = (z8 - parity of z1 + ... + z7) / 2; `mc` = 2 m + c
        const uint32_t odd = (z[0] ^ z[1] ^ z[2] ^ z[3] ^ z[4] ^ z[5] ^ z[6]) & 1u;
        const int32_t m2 = int32_t(z[7] - odd - 0x4B400000u);
        z[7] = 0x4B400000u + uint32_t(m2 >> 1);
        if (P.fields) {                                        // (0x4B400000 has no bits below 2^22: the low halves are the values')
            P.fields[here] = make_uint4(__byte_perm(z[0], z[1], 0x5410), __byte_perm(z[2], z[3], 0x5410), __byte_perm(z[4], z[5], 0x5410),
                                        __byte_perm(z[6], uint32_t(m2) + half, 0x5410));
        }
        ++blocks;
        halves += half;
        uint32_t *const column = hot + (half ? 8u * kHotStride : 0u) + lane;
        uint32_t far = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t u = min(z[j] - (0x4B400000u + uint32_t(kHotOrigin)), uint32_t(kHotBins));
            far |= u;
            atomicAdd(column + uint32_t(j) * kHotStride + u * 32u, 1u);
        }
        if (far & uint32_t(kHotBins)) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int32_t value = int32_t(z[j] - 0x4B400000u);
                if (uint32_t(value - kHotOrigin) >= uint32_t(kHotBins)) count_far(1u + 8u * half + uint32_t(j), value);
            }
        }
    }
    // the coset table
    blocks = warp_sum(blocks);
    halves = warp_sum(halves);
    if (lane == 0) {
        if (blocks != halves) atomicAdd(&win[0 - kWinOrigin], blocks - halves);
        if (halves) atomicAdd(&win[1 - kWinOrigin], halves);
    }
    __syncthreads();
    // columns into the window (two threads per value), then the window into global memory
    {
        const uint32_t bin = tid >> 1, t = bin / kHotBins, u = bin % kHotBins;
        static_assert(16u * kHotBins * 2u == kCountThreads, "two threads per value");
        uint32_t n = 0;
#pragma unroll
        for (uint32_t j = 0; j < 16; ++j) n += hot[t * kHotStride + u * 32u + ((j + (tid >> 1)) & 15u) + 16u * (tid & 1u)];
        if (n) atomicAdd(&win[(1u + t) * kWinBins + uint32_t(int32_t(u) + kHotOrigin - kWinOrigin)], n);
    }
    __syncthreads();
    static_assert(kWinBins % 32 == 0, "a warp's 32 counters are of one table");
    for (uint32_t j = tid; j < kWinWords; j += kCountThreads) {
        const uint32_t n = win[j], some = __ballot_sync(0xFFFFFFFFu, n != 0u);
        if (!some) continue;
        const uint32_t t = j / kWinBins, g = j % kWinBins + uint32_t(kWinOrigin - kHistOrigin), g0 = g - lane;
        if (n) atomicAdd(P.hist + (k * EP_NUM_TABLES + t) * kHistBins + g, n);
        if (lane == 0) {                         // the range of the 32: its first and last counter that is not zero
            atomicMax(&range_from[t], kHistBins - (g0 + uint32_t(__ffs(int(some)) - 1)));
            atomicMax(&range_to[t], g0 + 32u - uint32_t(__clz(int(some))));
        }
    }
    __syncthreads();
    if (tid < EP_NUM_TABLES && range_to[tid]) {
        atomicMax(&S.from[tid], range_from[tid]);
        atomicMax(&S.to[tid], range_to[tid]);
    }
    if (!arrive_last(&S.finished, ctas, last_cta)) return;
    const Evaluation E = gather_counts(P, k, P.mode == kPassSearch ? P.cand_counts + size_t(k) * kEvalSymbols : P.full_counts, sm, ranges);
    if (P.mode == kPassSearch) {
        __shared__ int32_t chosen;
        if (tid < 32u) {
            double rate;
            const uint32_t verdict = judge_candidate(P, k, E, rate);
            unsigned long long mine = 0, before = 0;
            if (lane == 1u) P.state->rate[k] = rate;
            __syncwarp();
            if (lane == 0) {
                S.overflow = 0;                                // (for the next pass)
                __threadfence();                               // the rate, and the counts, stored before gather_counts' last barrier
                mine = (static_cast<unsigned long long>(verdict) << (4u * k)) + (1ull << 60);
                before = atomicAdd(&P.state->verdicts, mine);
                __threadfence();
            }
            before = __shfl_sync(0xFFFFFFFFu, before + mine, 0);
            const int32_t last = (before >> 60) == scales ? take_steps(P, scales, before) : -1;
            if (lane == 0) chosen = last;
        }
        __syncthreads();
        if (chosen >= 0) keep_last(P, uint32_t(chosen));
        return;
    }
    if (tid < EP_NUM_TABLES) {
        P.state->full.lo[tid] = S.dir.lo[tid];
        P.state->full.K[tid] = S.dir.K[tid];
    }
    if (tid == 0) {
        if (__ldcg(&S.overflow)) P.state->overflow = 1;
        if (P.mode == kPassPolish) polish(P, s, E);
        const SearchState &G = *P.state;
        ended = P.entries && __ldcg(&G.polished) && __ldcg(&G.stop) && !__ldcg(&G.undecided) && !__ldcg(&G.overflow);
    }
    __syncthreads();
    if (ended) make_coder(P, sm, ranges);
}

// ---- Eq. 13: row scales ----------------------------------------------------------------------------------
__device__ __forceinline__ int32_t field16(uint32_t w, int hi) { return hi ? int32_t(w) >> 16 : int32_t(w << 16) >> 16; }
// 2 p of a block's eight weights (Eq. 5)
__device__ __forceinline__ void twice_point(const uint4 q, int32_t (&p2)[8]) {
    const int32_t mc = field16(q.w, 1), c = mc & 1;              // 2 m + c
    int32_t s7 = 0;
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        const int32_t z = field16(w[j >> 1], j & 1);
        s7 += z;
        p2[j] = 2 * z + c;
    }
    p2[7] = 2 * ((mc - c) + (s7 & 1)) + c;
}
__device__ __forceinline__ float refit_result(double xp, double pp, float s, float mu) {
    double sg;
    if (pp > 0.0) {
        sg = __ddiv_rn(xp, pp);
        if (!(sg > 1e-12)) sg = 1e-12;
    } else {
        sg = __dmul_rn(double(s), double(mu));
    }
    return __double2float_rn(sg);
}

// One row per CTA; see "sums over a row" above.  sum p^2 is exact in any order (multiples of 1/4 below 2^51).
__global__ void __launch_bounds__(kRowThreads) refit_kernel(const float *__restrict__ W, uint32_t C, const uint4 *__restrict__ fields,
                                                            float s, const SearchState *__restrict__ state, const float *__restrict__ mu,
                                                            float *__restrict__ sigma) {
    __shared__ double part[kRowThreads / 32];
    __shared__ __align__(16) float4 wbuf[2 * kRowThreads];
    __shared__ __align__(16) uint4 qbuf[kRowThreads];
    const uint32_t tid = threadIdx.x, per_row = C / 8;
    const float4 *x = reinterpret_cast<const float4 *>(W + size_t(blockIdx.x) * C);
    const uint4 *q = fields + size_t(blockIdx.x) * per_row;
    double xp = 0.0, pp4 = 0.0;                  // sum of x (2 p), sum of (2 p)^2
    float mag = 0.0f;                            // sum |x (2 p)|, to 1e-4
    for (uint32_t v = tid; v < per_row; v += kRowThreads) {
        const float4 a = __ldg(x + 2u * v), b = __ldg(x + 2u * v + 1u);
        int32_t p2[8], sq = 0;
        twice_point(__ldg(q + v), p2);
        const float xv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            xp = __fma_rn(double(xv[j]), double(p2[j]), xp);         // (38-bit products: exact)
            mag += fabsf(xv[j] * float(p2[j]));
            sq += p2[j] * p2[j];                                     // at most 8 * 2^26
        }
        pp4 = __dadd_rn(pp4, double(sq));
    }
    xp = 0.5 * cta_sum(xp, part);
    const double pp = 0.25 * cta_sum(pp4, part);
    const double off = order_bound(C, 0.501 * cta_sum(double(mag), part));
    if (state) s = state->s_counted;             // launched behind the search, before the host knows the scale
    const float m = __ldg(mu + blockIdx.x);
    const float lo = refit_result(__dsub_rn(xp, off), pp, s, m), hi = refit_result(__dadd_rn(xp, off), pp, s, m);
    // (launched while the tile coder runs, whose results it does not use; what is launched behind it, however, does)
    if (blockIdx.x == gridDim.x - 1u) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (lo == hi) {
        if (tid == 0) sigma[blockIdx.x] = lo;
        return;
    }
    xp = 0.0;                                    // index order
    for (uint32_t v0 = 0; v0 < per_row; v0 += kRowThreads) {
        __syncthreads();
        if (v0 + tid < per_row) {
            wbuf[2 * tid] = __ldg(x + 2u * (v0 + tid));
            wbuf[2 * tid + 1] = __ldg(x + 2u * (v0 + tid) + 1u);
            qbuf[tid] = __ldg(q + v0 + tid);
        }
        __syncthreads();
        if (tid == 0)
            for (uint32_t i = 0, n = min(kRowThreads, per_row - v0); i < n; ++i) {
                const float4 a = wbuf[2 * i], b = wbuf[2 * i + 1];
                int32_t p2[8];
                twice_point(qbuf[i], p2);
                const float xv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                for (int j = 0; j < 8; ++j) xp = __dadd_rn(xp, __dmul_rn(double(xv[j]), 0.5 * double(p2[j])));
            }
    }
    if (tid == 0) sigma[blockIdx.x] = refit_result(xp, pp, s, m);
}

// ---- tile coding (Sec. 3.6 / App. "Tiled rANS implementation", Eq. 17) ---------------------------------------
// (A kernel that comes up while the one before it runs takes that one's results by ordinary loads: __restrict__ and the
// read-only path promise that nobody writes the data while the kernel exists, and let a load move above the wait.)
__global__ void encode_entries_kernel(const uint32_t *fF, uint32_t n, uint32_t b, uint4 *entries) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    chained_start();
    if (i < n) entries[i] = encode_entry(fF[i], b);
}

// One warp per tile, one state per lane.  The decoder reads, per (group, field), the words of the needy lanes in
// ascending lane order; the encoder walks groups and fields backwards and fills the tile's word area from its end, writing
// each step's words as one block in ascending lane order, which is the order the reversed word list of a sequential
// encoder would have.  A step's chain is compare, shift, multiply-high, shift, multiply-add (about 30 cycles);
// a group's fields are asked for four groups ahead and its symbols looked up before the steps that need them.
// IN_SMEM: the symbols' entries in shared memory (up to 11 Ki symbols), else in global memory.  A CTA has four warps -
// tiles spread over the SMs - or sixteen where its table takes so much shared memory that few CTAs fit an SM.
constexpr uint32_t kTileThreads = 128, kTileThreadsMax = 512, kAhead = 4, kReportCtas = 8;

// A group's nine steps.  A step's words are stored during the next one: ballot, population counts and address (some 60 cycles)
// stay off the chain of states, and the store is predicated, not a branch.  P / Q: this and the previous step's
// predicate, B / C their ballots, H / I their states before the shift.
#define EP_CODE_LOAD(LD, J, A) LD " {a" J ", b" J ", c" J ", d" J "}, [" A "];\n\t"
#define EP_CODE_COUNT(C) "popc.b32 n, " C ";\n\t"  "and.b32 t, " C ", %3;\n\t"  "popc.b32 t, t;\n\t"
#define EP_CODE_STORE(Q, C, I)                                                                        \
    "sub.u32 %1, %1, n;\n\t"  "add.u32 t, t, %1;\n\t"  "mad.wide.u32 ad, t, 2, %2;\n\t"  "@" Q " st.global.u16 [ad], " I ";\n\t"
#define EP_CODE_STEP(J, P, B, H, COUNT, STORE)                                                        \
    COUNT "setp.ge.and.u32 " P ", %0, b" J ", act;\n\t"  "cvt.u16.u32 " H ", %0;\n\t"                        \
    "@" P " shr.u32 %0, %0, 16;\n\t"  "mul.hi.u32 q, %0, a" J ";\n\t"                                         \
    "vote.sync.ballot.b32 " B ", " P ", 0xffffffff;\n\t"  "shr.u32 o, d" J ", 16;\n\t"  "add.u32 o, o, %0;\n\t" \
    "shf.r.wrap.b32 q, q, 0, d" J ";\n\t"  "@act mad.lo.u32 %0, q, c" J ", o;\n\t" STORE
#define EP_CODE_REGS(J) ".reg .b32 a" J ", b" J ", c" J ", d" J ";\n\t"
#define EP_CODE_GROUP(LD, RT, A8, A7, A6, A5, A4, A3, A2, A1, A0)                                      \
    asm volatile("{\n\t.reg .pred act, pa, pb;\n\t.reg .b32 n, t, q, o, ba, bb;\n\t.reg .b16 ha, hb;\n\t.reg .b64 ad;\n\t"     \
        EP_CODE_REGS("8") EP_CODE_REGS("7") EP_CODE_REGS("6") EP_CODE_REGS("5") EP_CODE_REGS("4") EP_CODE_REGS("3") EP_CODE_REGS("2")   \
        EP_CODE_REGS("1") EP_CODE_REGS("0") "setp.ne.u32 act, %4, 0;\n\t"                                                        \
        EP_CODE_LOAD(LD, "8", "%5") EP_CODE_LOAD(LD, "7", "%6") EP_CODE_LOAD(LD, "6", "%7") EP_CODE_LOAD(LD, "5", "%8")               \
        EP_CODE_LOAD(LD, "4", "%9") EP_CODE_LOAD(LD, "3", "%10") EP_CODE_LOAD(LD, "2", "%11") EP_CODE_LOAD(LD, "1", "%12")           \
        EP_CODE_LOAD(LD, "0", "%13")                                                                                                \
        EP_CODE_STEP("8", "pa", "ba", "ha", "", "")                                                                                      \
        EP_CODE_STEP("7", "pb", "bb", "hb", EP_CODE_COUNT("ba"), EP_CODE_STORE("pa", "ba", "ha")) EP_CODE_STEP("6", "pa", "ba", "ha", EP_CODE_COUNT("bb"), EP_CODE_STORE("pb", "bb", "hb")) \
        EP_CODE_STEP("5", "pb", "bb", "hb", EP_CODE_COUNT("ba"), EP_CODE_STORE("pa", "ba", "ha")) EP_CODE_STEP("4", "pa", "ba", "ha", EP_CODE_COUNT("bb"), EP_CODE_STORE("pb", "bb", "hb")) \
        EP_CODE_STEP("3", "pb", "bb", "hb", EP_CODE_COUNT("ba"), EP_CODE_STORE("pa", "ba", "ha")) EP_CODE_STEP("2", "pa", "ba", "ha", EP_CODE_COUNT("bb"), EP_CODE_STORE("pb", "bb", "hb")) \
        EP_CODE_STEP("1", "pb", "bb", "hb", EP_CODE_COUNT("ba"), EP_CODE_STORE("pa", "ba", "ha")) EP_CODE_STEP("0", "pa", "ba", "ha", EP_CODE_COUNT("bb"), EP_CODE_STORE("pb", "bb", "hb")) \
        EP_CODE_COUNT("ba") EP_CODE_STORE("pa", "ba", "ha") "}"                                                                                          \
        : "+r"(x), "+r"(end) : "l"(area), "r"(lt), "r"(act), RT(A8), RT(A7), RT(A6), RT(A5), RT(A4), RT(A3), RT(A2), RT(A1), RT(A0) : "memory")

// The tables' place is in device memory: made by the pass that ended the search, or brought by the host.  A launch is for tables of more
// than `above` and at most `most` entries (which the host does not know yet when it launches) and does nothing else.
struct Report {                      // what `ctas` CTAs of the launch, behind those that code, bring to the host meanwhile
    uint32_t ctas;
    const uint32_t *last_counts, *full_counts, *full_freq;
    uint32_t *mail;                  // page-locked: as DeviceBackend's mail
};
struct TileParams {
    const uint4 *fields;
    uint32_t n_vec, V, n_tiles, cap, above, most;
    const uint4 *entries;
    uint16_t *scratch;
    uint32_t *index, *counts;
    SearchState *state;
    volatile uint64_t *total_words;  // page-locked: words of the payload (more than a blob can hold are still told apart)
    Report report;
};
constexpr size_t kMailLast = kStateBytes, kMailFull = kMailLast + 4ull * kEvalSymbols, kMailFreq = kMailFull + 4ull * EP_NUM_TABLES * kHistBins,
                 kMailDone = kMailFreq + 4ull * kMaxTableSymbols, kMailBytes = kMailDone + 64;      // done: u32 there, u32, u64 words

__device__ __noinline__ void report_search(const TileParams &P, uint32_t cta) {
    SearchState &S = *P.state;
    const uint32_t at = cta * blockDim.x + threadIdx.x, step = P.report.ctas * blockDim.x, lane = threadIdx.x & 31u;
    auto bring = [&](size_t to, const uint32_t *from, uint32_t n) {
#pragma unroll 8
        for (uint32_t i = at; i < n; i += step) P.report.mail[to / 4u + i] = __ldcg(from + i);
    };
    const uint32_t n_last = warp_sum(lane < EP_NUM_TABLES ? __ldcg(&S.last.K[lane]) : 0u), n_full = warp_sum(lane < EP_NUM_TABLES ? __ldcg(&S.full.K[lane]) : 0u);
    bring(0, reinterpret_cast<const uint32_t *>(&S), uint32_t(offsetof(SearchState, cand) / 4u));
    if (__ldcg(&S.has_last)) bring(kMailLast, P.report.last_counts, min(n_last, kEvalSymbols));
    bring(kMailFull, P.report.full_counts, n_full);
    if (__ldcg(&S.code)) bring(kMailFreq, P.report.full_freq, n_full);
    __syncthreads();
    if (threadIdx.x) return;
    __threadfence_system();          // (cumulative: the whole CTA's stores)
    if (atomicAdd(&S.reported, 1u) == P.report.ctas - 1u) {
        __threadfence_system();
        *const_cast<volatile uint32_t *>(P.report.mail + kMailDone / 4u) = 1u;
    }
}

template <bool IN_SMEM>
__global__ void __launch_bounds__(kTileThreadsMax) tile_encode_kernel(const __grid_constant__ TileParams P) {
    extern __shared__ __align__(16) uint4 entries_smem[];
    __shared__ uint32_t last_cta;
    __shared__ uint64_t part[kTileThreadsMax / 32];
    __shared__ EncodeTables tables;
    __shared__ uint32_t code;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, coders = gridDim.x - P.report.ctas;
    const uint32_t n_vec = P.n_vec, V = P.V, n_tiles = P.n_tiles, cap = P.cap;
    const uint4 *const fields = P.fields, *const entries_global = P.entries;
    uint16_t *const scratch = P.scratch;
    uint32_t *const index = P.index, *const counts = P.counts;
    SearchState *const state = P.state;
    chained_start();
    if (blockIdx.x >= coders) {
        report_search(P, blockIdx.x - coders);
        return;
    }
    if (tid < sizeof(EncodeTables) / 4u) reinterpret_cast<uint32_t *>(&tables)[tid] = __ldcg(reinterpret_cast<const uint32_t *>(&state->coder) + tid);
    if (tid == sizeof(EncodeTables) / 4u) code = __ldcg(&state->code);
    __syncthreads();
    EncodeTables T;                  // (by shuffles: known to be warp-uniform, see the warp's number below)
#pragma unroll
    for (int k = 0; k < 9; ++k) T.base[k] = __shfl_sync(0xFFFFFFFFu, tables.base[k], 0);
    T.coset = __shfl_sync(0xFFFFFFFFu, tables.coset, 0);
    T.total = __shfl_sync(0xFFFFFFFFu, tables.total, 0);
    if (!__shfl_sync(0xFFFFFFFFu, code, 0) || T.total <= P.above || T.total > P.most) return;
    if (IN_SMEM) {
        for (uint32_t i = tid; i < T.total; i += blockDim.x) entries_smem[i] = entries_global[i];
        __syncthreads();
    }
    const uint32_t entries = IN_SMEM ? uint32_t(__cvta_generic_to_shared(entries_smem)) : 0u;
    // (the warp's number by a shuffle: known to be warp-uniform, so no guard around the votes)
    const uint32_t tile = blockIdx.x * (blockDim.x >> 5) + __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    if (tile < n_tiles) {
        const uint32_t v0 = tile * V, nv = min(V, n_vec - v0), lt = (1u << lane) - 1u;
        const uint4 *const q = fields + v0;
        uint16_t *const area = scratch + size_t(tile) * cap;
        uint32_t end = cap;                      // words [end, cap) of the area are written
        uint32_t x = kStateLow;
        const uint32_t groups = (nv + 31u) >> 5;
        // Fields of the next groups on their way to shared memory, every lane its own 16 bytes: a group takes 0.2 us, a load
        // from L2 0.4.  (Loads into registers some groups ahead are waited for all together, the newest with the one
        // that is needed: 0.5 us per group.)
        const uint32_t staged = uint32_t(__cvta_generic_to_shared(entries_smem)) + (IN_SMEM ? 16u * T.total : 0u) + (tid >> 5) * (kAhead * 512u) + 16u * lane;
        auto ask = [&](uint32_t g) {             // group g, if there is one
            if (g < groups)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(staged + (g % kAhead) * 512u), "l"(q + min(g * 32u + lane, nv - 1u)) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (uint32_t i = 0; i < kAhead; ++i) ask(groups - 1u - i);
        for (uint32_t g = groups; g-- > 0;) {
            uint4 cur;
            asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1u) : "memory");
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(cur.x), "=r"(cur.y), "=r"(cur.z), "=r"(cur.w) : "r"(staged + (g % kAhead) * 512u) : "memory");
            ask(g - kAhead);                     // (past the first group: none, the number wraps)
            const int32_t mc = field16(cur.w, 1);
            const uint32_t w[4] = {cur.x, cur.y, cur.z, cur.w}, coset = (mc & 1) ? entries + T.coset : entries;
            uint32_t at[9];                      // (every offset is in range: these are the fields the tables were counted from)
            at[0] = T.base[0] + entries + 16u * uint32_t(mc & 1);
#pragma unroll
            for (int k = 1; k < 8; ++k) at[k] = 16u * uint32_t(field16(w[(k - 1) >> 1], (k - 1) & 1)) + (coset + T.base[k]);
            at[8] = 16u * uint32_t(mc >> 1) + (coset + T.base[8]);
            const uint32_t act = g * 32u + lane < nv ? 1u : 0u;      // a lane without a block keeps its state and gives off no word
            if (IN_SMEM) {
                EP_CODE_GROUP("ld.shared.v4.u32", "r", at[8], at[7], at[6], at[5], at[4], at[3], at[2], at[1], at[0]);
            } else {
                const uint64_t e0 = reinterpret_cast<uint64_t>(entries_global);
                EP_CODE_GROUP("ld.global.v4.u32", "l", e0 + at[8], e0 + at[7], e0 + at[6], e0 + at[5], e0 + at[4], e0 + at[3], e0 + at[2],
                              e0 + at[1], e0 + at[0]);
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        index[size_t(tile) * 33u + lane] = x;
        if (lane == 0) counts[tile] = cap - end;
    }
    // the last CTA turns the counts into offsets (the tile records' last words and the final one)
    if (!arrive_last(&state->tiles_done, coders, last_cta)) return;
    // (eight tiles per thread and turn, their loads under way together: one after another they took 0.7 us each, 16 us for 2743 tiles)
    const uint32_t warps = blockDim.x >> 5;
    uint64_t all = 0;
    for (uint32_t t0 = 0; t0 < n_tiles; t0 += 8u * blockDim.x) {
        const uint32_t t = t0 + 8u * tid;
        uint32_t n[8];
#pragma unroll
        for (uint32_t u = 0; u < 8u; ++u) n[u] = t + u < n_tiles ? __ldcg(counts + t + u) : 0u;
        uint64_t sum = 0;
#pragma unroll
        for (uint32_t u = 0; u < 8u; ++u) sum += n[u];
        uint64_t upto = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t before = __shfl_up_sync(0xFFFFFFFFu, upto, d);
            if (lane >= uint32_t(d)) upto += before;
        }
        if (lane == 31u) part[tid >> 5] = upto;
        __syncthreads();
        uint64_t at = all + upto - sum;
        for (uint32_t w = 0; w < warps; ++w) {
            if (w < tid >> 5) at += part[w];
            all += part[w];
        }
#pragma unroll
        for (uint32_t u = 0; u < 8u; ++u) {
            if (t + u < n_tiles) index[size_t(t + u) * 33u + 32u] = uint32_t(at);
            at += n[u];
        }
        __syncthreads();
    }
    if (tid == 0) {
        index[size_t(n_tiles) * 33u] = uint32_t(all);
        *P.total_words = all;
        state->tiles_done = 0;
    }
}

// Move every tile's words from the end of its area to its place in the payload: one CTA per tile (with a warp per tile the
// copy of 20 MB took 34 us, all of it waiting for loads; 19 so), four bytes per lane, the destination aligned.
__global__ void __launch_bounds__(512) compact_kernel(const uint16_t *scratch, uint32_t cap, const uint32_t *counts, const uint32_t *index,
                                                      const SearchState *state, uint16_t *payload) {
    const uint32_t tid = threadIdx.x, tile = blockIdx.x;
    chained_start();
    if (!__ldcg(&state->code)) return;           // nothing was coded
    uint32_t n = counts[tile];
    const uint16_t *src = scratch + size_t(tile) * cap + (cap - n);
    uint16_t *dst = payload + index[size_t(tile) * 33u + 32u];
    if (n && (reinterpret_cast<uintptr_t>(dst) & 2)) {
        if (tid == 0) *dst = *src;
        ++src; ++dst; --n;
    }
    uint32_t *const d32 = reinterpret_cast<uint32_t *>(dst);
    const uint32_t pairs = n / 2u;
    if (reinterpret_cast<uintptr_t>(src) & 2) {
        // each pair straddles two aligned words (the one before src starts inside the buffer, as src is not its start)
        const uint32_t *s32 = reinterpret_cast<const uint32_t *>(src - 1);
#pragma unroll 4
        for (uint32_t i = tid; i < pairs; i += blockDim.x) d32[i] = __funnelshift_r(s32[i], s32[i + 1u], 16);
    } else {
        const uint32_t *s32 = reinterpret_cast<const uint32_t *>(src);
#pragma unroll 4
        for (uint32_t i = tid; i < pairs; i += blockDim.x) d32[i] = s32[i];
    }
    if ((n & 1u) && tid == 0) dst[n - 1u] = src[n - 1u];
}

size_t align_up(size_t v) { return (v + 255) & ~size_t(255); }

struct Workspace {
    float *mu;
    uint32_t *rows, *hist, *counts, *fF, *cand_counts, *last_counts, *full_counts;
    SearchState *state;
    uint4 *entries;
    uint4 *fields;
    uint16_t *scratch;
    // the last three sections of the blob, back to back as they are stored: row scales, tile index, payload
    float *sigma;
    uint32_t *index;
    uint16_t *payload;
    size_t bytes;
};

constexpr size_t kHistBytes = 4ull * EP_NUM_TABLES * kHistBins;

Workspace carve(uint8_t *base, uint32_t R, uint32_t C, uint32_t V) {
    const uint64_t nvec = uint64_t(R) * (C / 8);
    const uint64_t n_tiles = (nvec + V - 1) / V;
    const uint64_t cap = 9ull * V;
    size_t at = 0;
    auto take = [&](size_t n) { uint8_t *p = base ? base + at : nullptr; at += align_up(n); return p; };
    Workspace w{};
    w.mu = reinterpret_cast<float *>(take(4ull * R));
    w.rows = reinterpret_cast<uint32_t *>(take(4ull * R));
    // state, then the counts of the last step, so that one copy brings both
    w.state = reinterpret_cast<SearchState *>(take(kStateBytes + 4ull * kEvalSymbols));
    w.last_counts = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(w.state) + kStateBytes);
    w.hist = reinterpret_cast<uint32_t *>(take(kCandidates * kHistBytes));
    w.cand_counts = reinterpret_cast<uint32_t *>(take(4ull * kCandidates * kEvalSymbols));
    w.full_counts = reinterpret_cast<uint32_t *>(take(kHistBytes));
    w.fF = reinterpret_cast<uint32_t *>(take(4ull * kCoderEntries));
    w.entries = reinterpret_cast<uint4 *>(take(16ull * kCoderEntries));
    w.counts = reinterpret_cast<uint32_t *>(take(4ull * n_tiles));
    w.fields = reinterpret_cast<uint4 *>(take(16ull * nvec));
    w.scratch = reinterpret_cast<uint16_t *>(take(2ull * cap * n_tiles + 4));
    uint8_t *tail = take(4ull * R + uint64_t(kTileRecordBytes) * n_tiles + 4 + 2ull * cap * n_tiles);
    w.sigma = reinterpret_cast<float *>(tail);
    if (base) {
        w.index = reinterpret_cast<uint32_t *>(tail + 4ull * R);
        w.payload = reinterpret_cast<uint16_t *>(tail + 4ull * R + uint64_t(kTileRecordBytes) * n_tiles + 4);
    }
    w.bytes = at;
    return w;
}

#define EP_CUDA(call)                                \
    do {                                             \
        if ((call) != cudaSuccess) return EP_ERR_CUDA; \
    } while (0)

// Page-locked host memory: for finished blobs and for the counts that come back after a search or a counting pass.
// Locking memory costs milliseconds, so each of the two uses keeps the buffer it last gave back (one at most, the
// larger one when two compete) for the next request that fits into it.
struct PinnedSlot {
    std::mutex lock;
    uint8_t *spare = nullptr;
    size_t spare_cap = 0;

    uint8_t *acquire(size_t n, size_t headroom, size_t *cap) {
        {
            std::lock_guard<std::mutex> hold(lock);
            if (spare && spare_cap >= n) {
                uint8_t *p = spare;
                *cap = spare_cap;
                spare = nullptr;
                spare_cap = 0;
                return p;
            }
        }
        const size_t want = n + headroom;
        void *p = nullptr;
        if (cudaHostAlloc(&p, want, cudaHostAllocDefault) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        *cap = want;
        return static_cast<uint8_t *>(p);
    }
    void release(uint8_t *p, size_t cap) {
        uint8_t *drop = p;
        {
            std::lock_guard<std::mutex> hold(lock);
            if (cap > spare_cap) {               // keep the larger of the two
                drop = spare;
                spare = p;
                spare_cap = cap;
            }
        }
        if (drop) cudaFreeHost(drop);
    }
};
PinnedSlot g_blob_slot, g_mail_slot;

// headroom for blobs: the next tensor of a model is rarely the same size
uint8_t *pinned_acquire(size_t n, size_t *cap) { return g_blob_slot.acquire(n, n / 8 + 4096, cap); }
void pinned_release(uint8_t *p, size_t cap) { g_blob_slot.release(p, cap); }

class DeviceBackend final : public EncodeBackend {
public:
    DeviceBackend(const float *dW, uint32_t R, uint32_t C, uint32_t V, uint8_t *ws, cudaStream_t st)
        : W_(dW), R_(R), C_(C), V_(V), w_(carve(ws, R, C, V)), st_(st) {
        mail_ = g_mail_slot.acquire(kMailBytes, 0, &mail_cap_);
        if (!mail_) throw std::bad_alloc();
    }
    ~DeviceBackend() override {
        // a call that ends early must not leave a copy into the page-locked buffers behind, which the next call may have then
        if (under_way_) cudaStreamSynchronize(st_);
        if (mail_) g_mail_slot.release(mail_, mail_cap_);
    }

    int prepare(const std::vector<uint32_t> &sample) override {
        n_sample_ = uint32_t(sample.size());
        under_way_ = true;
        int dev = 0;
        EP_CUDA(cudaGetDevice(&dev));
        EP_CUDA(cudaDeviceGetAttribute(&sms_, cudaDevAttrMultiProcessorCount, dev));
        EP_CUDA(cudaFuncSetAttribute(quantise_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kCountSmem)));
        // (a sample of all rows, as smaller tensors have it, needs no list)
        sample_rows_ = n_sample_ < R_ ? w_.rows : nullptr;
        if (sample_rows_) EP_CUDA(cudaMemcpyAsync(w_.rows, sample.data(), 4ull * n_sample_, cudaMemcpyHostToDevice, st_));
        // the state, and the histograms behind it (every pass leaves them zero again)
        const size_t clear = size_t(reinterpret_cast<uint8_t *>(w_.hist) - reinterpret_cast<uint8_t *>(w_.state)) + kCandidates * kHistBytes;
        row_rms_kernel<<<R_ + kClearCtas, kRowThreads, 0, st_>>>(W_, C_, w_.mu, reinterpret_cast<uint4 *>(w_.state), uint32_t(clear / 16u));
        EP_CUDA(cudaGetLastError());
        state_clear_ = true;
        return EP_OK;
    }
    int count_sample(float s, Model &m) override { return count(sample_rows_, n_sample_, s, nullptr, m); }
    int count_full(float s, Model &m) override { return count(nullptr, R_, s, w_.fields, m); }

    int search(const SearchJob &job, const ep_encode_opts &o, SearchResult &r, bool *done) override {
        *done = false;
        if (!state_clear_) EP_CUDA(cudaMemsetAsync(w_.state, 0, kStateBytes, st_));
        state_clear_ = false;
        // with the refinement of rows (which this back end leaves to the host) the last pass's tables are not the final ones
        const bool ahead = o.rdo_candidates <= 1;
        CountParams P = params(sample_rows_, n_sample_, 0.0f, nullptr);
        P.mode = kPassSearch;
        P.rate = rate_params(job.target_bpp, o.retained_bits, job.sample_vectors, job.sample_rows, job.V, job.b);
        P.lo0 = o.bracket_lo;
        P.hi0 = o.bracket_hi;
        const float s0 = float(std::sqrt(o.bracket_lo * o.bracket_hi));
        if (o.search_steps == 0) EP_CUDA(cudaMemcpyAsync(&w_.state->s, &s0, 4, cudaMemcpyHostToDevice, st_));
        // the first step, then passes of several scales: as many as the steps take four at a time, and one that the forecast may lose.
        // Up to 2^17 blocks fifteen scales cost little more than nine, beyond it they do
        P.steps = uint32_t(o.search_steps);
        P.most = P.n_blocks <= (1u << 17) ? kCandidates : 9u;
        const uint32_t passes = o.search_steps < 2 ? uint32_t(o.search_steps) : 2u + (P.steps - 1u + kLevels - 1u) / kLevels;
        for (uint32_t pass = 0; pass < passes; ++pass) {
            P.pass = pass;
            P.after = passes - std::min(passes, pass + 2u);
            EP_CUDA(launch_count(P, pass > 0));
        }
        CountParams F = params(nullptr, R_, 0.0f, w_.fields);
        F.mode = kPassPolish;
        F.rate = rate_params(job.target_bpp, o.polish_retained_bits, F.n_blocks, R_, job.V, job.b);
        F.lo0 = o.bracket_lo;
        F.hi0 = o.bracket_hi;
        F.last_step = o.polish_steps;
        F.entries = ahead ? w_.entries : nullptr;
        F.full_freq = w_.fF;
        for (F.step = 0;; ++F.step) {
            EP_CUDA(launch_count(F, F.step > 0 || o.search_steps > 0));
            if (F.step == o.polish_steps) break;
            if (F.step % 8 == 7) {               // a caller may allow any number of corrections: is there still something to correct?
                EP_CUDA(cudaMemcpyAsync(&state()->stop, &w_.state->stop, sizeof(state()->stop), cudaMemcpyDeviceToHost, st_));
                EP_CUDA(cudaStreamSynchronize(st_));
                if (state()->stop) break;
            }
        }
        int rc = EP_OK;
        if (ahead) {
            // The tiles are coded and the row scales made without waiting for the host, which meanwhile makes its own tables of the same
            // counts.  If the search goes on on the host, what was coded is not used.  Whole encode, copied back, with the clearing in
            // row_rms_kernel and the faster prefix sum of the tiles: 10240 x 3840 at 4 bpp 1249 -> 1209 us, 512 x 1024 240 -> 222.
            // The refit runs beside the tile coder: one after the other they took 109 us for 10240 x 3840, together 90.
            std::memset(mail_ + kMailDone, 0, kMailBytes - kMailDone);
            const uint32_t n_tiles = uint32_t((uint64_t(R_) * (C_ / 8) + V_ - 1) / V_);
            EP_CUDA(launch_coder(n_tiles, 0u, kFewEntries, true));
            EP_CUDA(launch_beside(refit_kernel, R_, kRowThreads, 0, W_, C_, static_cast<const uint4 *>(w_.fields), 0.0f, static_cast<const SearchState *>(w_.state),
                                   static_cast<const float *>(w_.mu), w_.sigma));
            EP_CUDA(launch_coder(n_tiles, kFewEntries, kSmemEntries, false));
            EP_CUDA(launch_compact(n_tiles));
            rc = await_report();
        } else {
            rc = fetch(true);
            if (!rc) refit_kernel<<<R_, kRowThreads, 0, st_>>>(W_, C_, w_.fields, 0.0f, w_.state, w_.mu, w_.sigma);
            EP_CUDA(cudaGetLastError());
        }
        if (rc) return rc;
        const SearchState &S = *state();
        if (S.undecided || S.left) {             // (steps left: cannot happen, and the scale would not be the bisection's)
            EP_CUDA(cudaMemsetAsync(w_.state, 0, kStateBytes, st_));
            return EP_OK;
        }
        coded_ = ahead && S.code && *reported();      // (without the report the frequencies to compare are not here)
        coded_b_ = job.b;
        r.s = sigma_of_ = S.s_counted;
        sigma_there_ = true;
        r.polished = S.polished != 0;
        r.has_last = S.has_last != 0;
        if (r.has_last) r.last.from_counts(S.last.lo, S.last.K, last_counts());
        r.full.from_counts(S.full.lo, S.full.K, full_counts());
        *done = true;
        return EP_OK;
    }

    int begin_finish(float s, int b, uint32_t V, const Model &m) override {
        const uint64_t nvec = uint64_t(R_) * (C_ / 8);
        const uint32_t n_tiles = uint32_t((nvec + V - 1) / V);
        uint64_t symbols = 0;
        for (int t = 0; t < EP_NUM_TABLES; ++t) symbols += m.t[t].K();
        if (symbols > kMaxTableSymbols) return EP_ERR_UNSUPPORTED;
        if (coded_ && sigma_there_ && sigma_of_ == s && coded_b_ == b && V == V_ && coded_with(m)) return EP_OK;
        const CoderLayout L = coder_layout(m);
        if (L.entries() > kCoderEntries) return EP_ERR_UNSUPPORTED;      // (no count lies outside the histogram: cannot happen)
        const uint32_t size = L.size;
        EncodeTables T{};
        T.coset = 16u * size;
        T.total = L.entries();
        std::vector<uint32_t> fF(T.total, 0);
        for (int k = 1; k < 9; ++k) {
            T.base[k] = 16u * (L.first[k] - uint32_t(L.lo[k]));
            for (int c = 0; c < 2; ++c) {
                const Table &tb = m.t[table_id(c, k)];
                if (!tb.K()) continue;
                uint32_t *to = fF.data() + uint32_t(c) * size + L.first[k] + uint32_t(tb.lo - L.lo[k]);
                for (uint32_t j = 0; j < tb.K(); ++j) to[j] = tb.f[j] | (tb.F[j] << 16);
            }
        }
        T.base[0] = 32u * size;                  // the coset's two entries last
        for (uint32_t j = 0; j < m.t[0].K(); ++j) fF[2u * size + uint32_t(m.t[0].lo) + j] = m.t[0].f[j] | (m.t[0].F[j] << 16);
        EP_CUDA(cudaMemcpyAsync(w_.fF, fF.data(), 4ull * fF.size(), cudaMemcpyHostToDevice, st_));
        struct { EncodeTables T; uint32_t code, tiles_done; } coder = {T, 1u, 0u};
        static_assert(offsetof(SearchState, code) == offsetof(SearchState, coder) + sizeof(EncodeTables) &&
                      offsetof(SearchState, tiles_done) == offsetof(SearchState, code) + 4, "one copy");
        EP_CUDA(cudaMemcpyAsync(&w_.state->coder, &coder, sizeof(coder), cudaMemcpyHostToDevice, st_));
        std::memset(mail_ + kMailDone, 0, kMailBytes - kMailDone);
        EP_CUDA(launch_chained(encode_entries_kernel, (T.total + 127u) / 128u, 128, 0, w_.fF, T.total, uint32_t(b), w_.entries));
        if (T.total <= kFewEntries) EP_CUDA(launch_coder(n_tiles, 0u, kFewEntries, false));
        else if (T.total <= kSmemEntries) EP_CUDA(launch_coder(n_tiles, kFewEntries, kSmemEntries, false));
        else EP_CUDA(launch_coder(n_tiles, kSmemEntries, ~0u, false));
        EP_CUDA(launch_compact(n_tiles));
        if (!sigma_there_ || sigma_of_ != s) refit_kernel<<<R_, kRowThreads, 0, st_>>>(W_, C_, w_.fields, s, nullptr, w_.mu, w_.sigma);
        EP_CUDA(cudaGetLastError());
        return EP_OK;
    }
    int end_finish(float s, int b, uint32_t V, const Model &m, double cce, ep_blob *out) override {
        const uint64_t nvec = uint64_t(R_) * (C_ / 8), n_tiles = (nvec + V - 1) / V;
        // how many words the tiles have is known when the device is done; the copy is issued now, for a few more than that.  Were they
        // more even so, the blob is laid out again
        const uint64_t before = kHeaderBytes + m.section_bytes() + 4ull * R_ + uint64_t(kTileRecordBytes) * n_tiles + 4u;
        uint64_t room = payload_room(cce, n_tiles, 9ull * V * n_tiles, before);
        if (!room) return EP_ERR_UNSUPPORTED;
        out->acquire = pinned_acquire;
        out->release = pinned_release;
        for (;;) {
            // header and tables are laid out on the host; the other sections are copied straight into their place
            BlobLayout L;
            const int rc = begin_blob(m, R_, C_, b, V, s, room, out, &L);
            if (rc) return rc;
            EP_CUDA(cudaMemcpyAsync(out->data() + L.off_scales, w_.sigma, L.total - L.off_scales, cudaMemcpyDeviceToHost, st_));
            EP_CUDA(cudaStreamSynchronize(st_));
            const uint64_t total = *total_words();
            if (total >= (1ull << 31)) return EP_ERR_UNSUPPORTED;
            if (total <= room) {
                under_way_ = false;
                end_blob(L, total, out);
                return EP_OK;
            }
            room = total;
        }
    }

private:
    // mail: state, counts of the last step, counts and frequencies of the full pass, what kernels write there themselves
    SearchState *state() { return reinterpret_cast<SearchState *>(mail_); }
    uint32_t *last_counts() { return reinterpret_cast<uint32_t *>(mail_ + kMailLast); }
    uint32_t *full_counts() { return reinterpret_cast<uint32_t *>(mail_ + kMailFull); }
    volatile uint32_t *reported() { return reinterpret_cast<volatile uint32_t *>(mail_ + kMailDone); }
    volatile uint64_t *total_words() { return reinterpret_cast<volatile uint64_t *>(mail_ + kMailDone + 8); }
    // the device's frequencies are the model's
    bool coded_with(const Model &m) const {
        const uint32_t *f = reinterpret_cast<const uint32_t *>(mail_ + kMailFreq);
        for (const Table &t : m.t) {
            if (t.f.size() != t.K() || std::memcmp(f, t.f.data(), 4ull * t.K())) return false;
            f += t.K();
        }
        return true;
    }
    // Tile coder for tables of more than `above` and at most `most` entries.  Few entries: four warps per CTA while the tiles then fit the
    // SMs at once (five such CTAs per SM), else eight, four times, or sixteen, three times
    cudaError_t launch_coder(uint32_t n_tiles, uint32_t above, uint32_t most, bool report) {
        const bool in_smem = most <= kSmemEntries;
        uint32_t threads = kTileThreads;
        if (in_smem) threads = most > kFewEntries || n_tiles > 32u * uint32_t(sms_) ? kTileThreadsMax : n_tiles > 20u * uint32_t(sms_) ? 2u * kTileThreads : kTileThreads;
        const size_t stage = kAhead * 512u, smem = threads / 32u * stage + (in_smem ? 16ull * most : 0u);
        TileParams P{};
        P.fields = w_.fields;
        P.n_vec = uint32_t(uint64_t(R_) * (C_ / 8));
        P.V = V_;
        P.n_tiles = n_tiles;
        P.cap = 9u * V_;
        P.above = above;
        P.most = most;
        P.entries = w_.entries;
        P.scratch = w_.scratch;
        P.index = w_.index;
        P.counts = w_.counts;
        P.state = w_.state;
        P.total_words = total_words();
        if (report) P.report = {kReportCtas, w_.last_counts, w_.full_counts, w_.fF, reinterpret_cast<uint32_t *>(mail_)};
        if (smem > 40u * 1024u) {    // (always the same limit: another thread's call must not lower it before the launch)
            const cudaError_t e = cudaFuncSetAttribute(tile_encode_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       int(16u * kSmemEntries + kTileThreadsMax / 32u * (kAhead * 512u)));
            if (e != cudaSuccess) return e;
        }
        const uint32_t ctas = (n_tiles + threads / 32u - 1u) / (threads / 32u) + P.report.ctas;
        // Behind a counting pass not while that still runs: its CTAs leave an SM no registers for others, so the first SMs it leaves would get
        // all coding CTAs of a small tensor (512 x 1024: 30 - 50 us instead of 20)
        if (report) {
            tile_encode_kernel<true><<<ctas, threads, smem, st_>>>(P);
            return cudaGetLastError();
        }
        return in_smem ? launch_chained(tile_encode_kernel<true>, ctas, threads, smem, P) : launch_chained(tile_encode_kernel<false>, ctas, threads, smem, P);
    }
    // (few CTAs: more threads per tile.  Whole encode, us, 512 / 128 threads: 37 tiles 247.4 / 251.0, 289 346.1 / 348.3, 577 397.8 / 397.9,
    // 1153 528.5 / 528.1, 2305 at 8 bpp 836.9 / 829.1, 4610 1320.7 / 1310.6)
    cudaError_t launch_compact(uint32_t n_tiles) {
        return launch_chained(compact_kernel, n_tiles, n_tiles < 600u ? 512u : 128u, 0, static_cast<const uint16_t *>(w_.scratch), 9u * V_,
                              static_cast<const uint32_t *>(w_.counts), static_cast<const uint32_t *>(w_.index), static_cast<const SearchState *>(w_.state), w_.payload);
    }
    // Until the search's report is here (report_search).  If that takes longer than 5 ms - a very large tensor, earlier work on the stream - the
    // stream's own end is waited for, in the way that the process has its threads wait: an error shows there, and a report that still
    // is not here is fetched.  (The host's tables then come behind the coder: some 40 us of a long call.)
    int await_report() {
        const auto since = std::chrono::steady_clock::now();
        for (uint32_t i = 1; !*reported(); ++i) {
            if (i % 1024u == 0 && std::chrono::steady_clock::now() - since > std::chrono::milliseconds(5)) {
                EP_CUDA(cudaStreamSynchronize(st_));
                if (!*reported()) return fetch(true);
                break;
            }
#if defined(__x86_64__)
            __builtin_ia32_pause();
#endif
        }
        std::atomic_thread_fence(std::memory_order_acquire);
        return state()->overflow && !state()->undecided ? EP_ERR_UNSUPPORTED : EP_OK;     // a coordinate beyond +-4095: use the host encoder
    }

    CountParams params(const uint32_t *rows, uint32_t n_rows, float s, uint4 *fields) {
        CountParams P{};
        P.W = W_;
        P.mu = w_.mu;
        P.rows = rows;
        P.fields = fields;
        P.hist = w_.hist;
        P.state = w_.state;
        P.last_counts = w_.last_counts;
        P.full_counts = w_.full_counts;
        P.cand_counts = w_.cand_counts;
        P.per_row = C_ / 8;
        P.n_blocks = n_rows * P.per_row;
        P.C = C_;
        P.mode = kPassCount;
        P.s = s;
        return P;
    }
    static RateParams rate_params(double target, double retained, uint64_t n, uint64_t rows, uint32_t V, int b) {
        const double tiles = double((n + V - 1) / V);
        return {target, retained * double(kStates) * tiles, tiles * (32.0 * kStates + 32.0) + 32.0 + 32.0 * double(rows) + 8.0 * kHeaderBytes,
                8.0 * double(n), 9.0 * double(n), b};
    }
    // launched while the kernel before it ends; the kernel waits on the device (chained_start)
    template <class... K, class... A>
    cudaError_t launch_chained(void (*kernel)(K...), uint32_t grid, uint32_t threads, size_t smem, A... args) {
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st_;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, K(args)...);
    }
    // Launched while the kernel before it runs, whose results it does not use, so the kernel does its work without waiting.  But what is launched behind
    // it, and only waits for it, may use them: one of its CTAs has to wait all the same before it ends (refit_kernel: the last)
    template <class... K, class... A>
    cudaError_t launch_beside(void (*kernel)(K...), uint32_t grid, uint32_t threads, size_t smem, A... args) {
        return launch_chained(kernel, grid, threads, smem, args...);
    }
    // one CTA per SM, each with at least a few hundred blocks
    cudaError_t launch_count(CountParams P, bool follows) {
        const bool listed = P.mode == kPassSearch && P.pass > 0u;
        const uint32_t ctas = listed ? pass_grid(uint32_t(sms_)) : std::max(1u, std::min((P.n_blocks + 255u) / 256u, uint32_t(sms_)));
        // A pass's last CTA works on alone for 8 us; with programmatic launch the next pass's CTAs come up meanwhile, load
        // their first blocks and clear their counters.  Not the first pass: it reads what the kernel before it writes.
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(kCountThreads);
        cfg.dynamicSmemBytes = kCountSmem;
        cfg.stream = st_;
        cfg.attrs = &attr;
        cfg.numAttrs = follows ? 1u : 0u;
        return cudaLaunchKernelEx(&cfg, quantise_count_kernel, P);
    }
    static size_t symbols(const CountDir &D) {
        size_t n = 0;
        for (uint32_t k : D.K) n += k;
        return n;
    }
    // state and counts to the host: most alphabets fit the first copy
    int fetch(bool last) {
        EP_CUDA(cudaMemcpyAsync(mail_, w_.state, kStateBytes + (last ? 4ull * kFirstCounts : 0), cudaMemcpyDeviceToHost, st_));
        EP_CUDA(cudaMemcpyAsync(full_counts(), w_.full_counts, 4ull * kFirstCounts, cudaMemcpyDeviceToHost, st_));
        EP_CUDA(cudaStreamSynchronize(st_));
        const SearchState &S = *state();
        // (after a step it could not decide a search may have gone where the host's does not)
        if (S.overflow && !(last && S.undecided)) return EP_ERR_UNSUPPORTED;     // a coordinate beyond +-4095: use the host encoder
        bool more = false;
        auto rest = [&](uint32_t *to, const uint32_t *from, size_t n) {
            if (n <= kFirstCounts) return cudaSuccess;
            more = true;
            return cudaMemcpyAsync(to + kFirstCounts, from + kFirstCounts, 4ull * (n - kFirstCounts), cudaMemcpyDeviceToHost, st_);
        };
        if (last && S.has_last) EP_CUDA(rest(last_counts(), w_.last_counts, symbols(S.last)));
        EP_CUDA(rest(full_counts(), w_.full_counts, symbols(S.full)));
        if (more) EP_CUDA(cudaStreamSynchronize(st_));
        return EP_OK;
    }
    int count(const uint32_t *rows, uint32_t n_rows, float s, uint4 *fields, Model &m) {
        EP_CUDA(launch_count(params(rows, n_rows, s, fields), false));
        sigma_there_ = false;
        const int rc = fetch(false);
        if (rc) return rc;
        m.from_counts(state()->full.lo, state()->full.K, full_counts());
        return EP_OK;
    }

    const float *W_;
    uint32_t R_, C_, V_;
    Workspace w_;
    cudaStream_t st_;
    int sms_ = 0;
    uint8_t *mail_ = nullptr;        // page-locked: the copies back are plain DMA
    size_t mail_cap_ = 0;
    uint32_t n_sample_ = 0;
    const uint32_t *sample_rows_ = nullptr;      // null: all rows
    bool under_way_ = false;         // the stream may still work for this call
    bool sigma_there_ = false;       // w_.sigma holds the row scales of the kept quantisation, which is at scale sigma_of_
    float sigma_of_ = 0.0f;
    bool state_clear_ = false;       // the search's state is zero
    bool coded_ = false;             // the tiles are coded (or being coded) from the counts of the last search, at precision
    int coded_b_ = 0;
};

uint32_t tile_vectors_of(const ep_encode_opts &o, double target_bpp) {
    return o.tile_vectors ? o.tile_vectors : ep_default_tile_vectors(target_bpp);
}

}  // namespace

extern "C" size_t ep_encode_device_workspace_bytes(uint32_t R, uint32_t C, double target_bpp, const ep_encode_opts *opts_in) {
    ep_encode_opts o;
    if (opts_in) o = *opts_in; else ep_encode_opts_default(&o);
    if (ep::check_encode_args(R, C, target_bpp, o)) return 0;
    return carve(nullptr, R, C, tile_vectors_of(o, target_bpp)).bytes;
}

extern "C" int ep_encode_device(const float *d_W, uint32_t R, uint32_t C, double target_bpp, const ep_encode_opts *opts_in,
                                void *d_workspace, size_t workspace_bytes, void *stream, ep_blob **out) {
    if (!d_W || !out || !d_workspace) return EP_ERR_BAD_ARG;
    ep_encode_opts o;
    if (opts_in) o = *opts_in; else ep_encode_opts_default(&o);
    const int bad = ep::check_encode_args(R, C, target_bpp, o);
    if (bad) return bad;
    if ((reinterpret_cast<uintptr_t>(d_W) & 15) || (reinterpret_cast<uintptr_t>(d_workspace) & 255)) return EP_ERR_BAD_ARG;
    const uint32_t V = tile_vectors_of(o, target_bpp);
    if (uint64_t(V) * 9u >= (1ull << 31) || uint64_t(R) * (C / 8) >= (1ull << 31)) return EP_ERR_UNSUPPORTED;
    if (workspace_bytes < carve(nullptr, R, C, V).bytes) return EP_ERR_SCRATCH;
    try {
        DeviceBackend be(d_W, R, C, V, static_cast<uint8_t *>(d_workspace), static_cast<cudaStream_t>(stream));
        return ep::run_encode(be, R, C, target_bpp, o, out);
    } catch (const std::bad_alloc &) {
        return EP_ERR_NOMEM;
    } catch (...) {
        return EP_ERR_UNSUPPORTED;
    }
}

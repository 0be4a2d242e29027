// Fused EntroPack decode for sm_100a (paper Sec. 3.7): tiled 32-state rANS symbol decode (Eq. 18),
// arithmetic inverse of the field representation (Eq. 5), multiplication by the fp32 row scale and
// rounding to the output type (Eq. 19), written straight to the weight tensor.  No symbol tensor,
// no codebook, no tensor cores (the path is not a contraction).
//
// Mapping: one warp per tile, one rANS state per lane (the paper's layout).  A CTA of 32 warps builds (or
// copies) the sixteen slot -> (frequency, offset, value) lookup tables of the coordinate fields once in
// shared memory and then streams tiles through them.  A lookup entry is one word
//     [31:21] f      [20:11] code     [10:0] u - F
// where `code` is the symbol's coordinate relative to an even base zlo (z - zlo; 2m - zlo for the m
// field).  f < 2^11 always: a coordinate table with a single symbol at b = 11 (f = 2^11) goes to the
// large-table path.  (entry & 0x1FF800) | 0x45800000 is the fp32 number 4096 + code (| 0x400 adds the
// half of coset 1), so one subtraction of 4096 - zlo yields the lattice coordinate p exactly, and one fp32
// multiply by the row scale gives the product of Eq. 19 with the same operands and rounding as the
// definition.  The coset symbol has two values only: it is decoded by comparing the slot with the
// frequency of coset 0, without a table.
//
// Payload words reach the lanes through a per-tile ring in shared memory, filled 512 bytes at a time by
// cp.async (16 bytes per lane, source clamped to the end of the payload) ahead of the read cursor; the
// first 512 bytes of the ring are mirrored behind its end so that the nine steps of a group never have
// to wrap an address.  (With b <= 11 a lane takes at most seven words in nine steps: a step shortens the
// state by at most eleven bits, a word adds sixteen.)
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "stream.hpp"

namespace {

// A warp decodes one tile at a time.  Two, three or four with their instructions interleaved and 24, 16 or 12 warps were slower
// (8192 x 8192 at 4 bpp to FP16 / the 372 M-parameter layer at 3.5 bpp to BF16, Gparams/s: 32 warps with one 985 / 1171, 24 with two
// 940 / 1104, 16 with three 781 / 889, 12 with four 677 / 744): the loop is bound by the issue slots, the ALU pipe and the
// shared-memory pipe together (each about 70 % busy), not by the latency of one tile's chain of steps.
constexpr int kWarps = 32;                                   // warps per CTA (one CTA per SM)
constexpr int kThreads = kWarps * 32;
constexpr uint32_t kTilesPerRound = kWarps;                  // tiles per CTA at a time, at most (see split_rounds)
// Most tiles per CTA for decode_tile_few: its 512 threads may use 128 registers.  1792-block tiles at 4 bpp to BF16, us, this
// loop / the ordinary one: 4 tiles 33.3 / 40.0, 8: 36.7 / 41.3, 12: 41.4 / 43.8, 16: 45.2 / 46.6.
constexpr uint32_t kFewTiles = 16;
constexpr uint32_t kMinWarps = 8;                            // warps of a CTA, however few tiles it has
// ... that builds its tables itself: a warp per table (1024 x 1024 at 6 bpp in tiles of 64 blocks, no prepared image, us: 8 warps
// 13.3, 16 warps 9.8).
constexpr uint32_t kBuildWarps = EP_NUM_TABLES - 1;
static_assert(kTilesPerRound == ep::kDecodeTilesPerCta, "tile-size suggestions assume this many tiles per CTA");
constexpr uint32_t kLutEntries = 2048;                       // 2^11 slots per table
constexpr uint32_t kLutStride = kLutEntries * 4;             // bytes per table in shared memory
constexpr uint32_t kCosetStride = 8 * kLutStride;            // the eight tables of coset 1 follow those of coset 0
constexpr uint32_t kLutBytes = 16 * kLutStride;              // 131072
// Payload ring of a tile: three chunks of 512 bytes (one cp.async round of a warp, 16 bytes per lane) plus a mirror
// of its first 512 bytes.  (Measured and dropped: 64 rings of four 256-byte chunks for two tiles per warp at 32 warps.)
constexpr uint32_t kChunk = 512, kRingSlots = 3;
constexpr uint32_t kRingBytes = kRingSlots * kChunk;         // 1536
constexpr uint32_t kRingMirror = 512;                        // >= 7 words * 32 lanes * 2 bytes + one lane span (62)
constexpr uint32_t kRingStride = kRingBytes + kRingMirror;   // 2048 per warp
constexpr uint32_t kCtxBytes = 64;                           // per warp: what the rare paths of the hot loop need
constexpr uint32_t kCtxBase = kLutBytes;
constexpr uint32_t kRingBase = kCtxBase + kWarps * kCtxBytes;
// 2^12-slot streams: per table, the entries of the kHotSpan coordinate values around zero are kept in shared memory
// (the rest is read from global memory); this fills what the tables, rings and context blocks
// leave of the 227 KB
constexpr uint32_t kHotSpan = 528;                           // coordinate codes per table in the hot window
constexpr uint32_t kHotBytes = 16 * kHotSpan * 4;            // 33792
constexpr uint32_t kColdCodes = 4096;                        // codes per table in the complete entry array (global memory)
constexpr uint32_t kColdBytes = 16 * kColdCodes * 4;         // 262144
constexpr uint32_t kHotBase = kRingBase + kWarps * kRingStride;
constexpr uint32_t kSmemBytes = kHotBase + kHotBytes;          // 232448
static_assert(kSmemBytes <= 232448, "more shared memory than an sm_100 CTA can have");
constexpr uint32_t kStageBytes = kSmemBytes - kRingBase;     // with few tiles per CTA: room for their whole payloads (see decode_tile_few)
constexpr uint32_t kCodeMask = 0x001FF800u;                  // 10-bit code field
constexpr uint32_t kExp4096 = 0x45800000u;                   // fp32 bit pattern of 4096.0
constexpr uint32_t kOwnSlots = 16;                           // table build: slots of a symbol that its own lane writes
constexpr uint32_t kEntryUnused = 1u << 21;                  // f = 1: what a slot no symbol owns holds (damaged tables)

// per-warp context block (byte offsets): the job's part, and the tile's from kCtxChain on
constexpr uint32_t kCtxScales = 0;         // u64 row scales
constexpr uint32_t kCtxRowBytes = 8;       // u32 output bytes per row
constexpr uint32_t kCtxRowMax = 12;        // u32 last row index
constexpr uint32_t kCtxTablesBar = 16;     // u64 mbarrier of the table image's copy (warp j's: of job j's, see ep_decode_smem_kernel)
constexpr uint32_t kCtxRowRcp = 24;        // u32 ceil(2^32 / bytes per row)
constexpr uint32_t kCtxChain = 32;
constexpr uint32_t kCcSrc = 0;             // u64 global address of lane 0's 16 bytes of the next chunk to request
constexpr uint32_t kCcRem = 8;             // s32 payload bytes from there to the end of the payload (may be <= 0)
constexpr uint32_t kCcDst = 12;            // u32 ring address of lane 0's 16 bytes of that chunk's slot
constexpr uint32_t kCcRing = 16;           // u32 ring base (shared-memory address)
constexpr uint32_t kCcWbase = 20;          // u32 ring address of byte position 0 (cursor address minus position)
constexpr uint32_t kCcEndo = 24;           // u32 output byte offset after the tile's last block

__device__ unsigned int g_ep_status = 0;

struct JobParams {
    const uint8_t *stream;        // blob base (device)
    const uint32_t *tile_index;   // n_tiles records of 33 words + 1 final word
    const float *scales;
    void *out;
    const uint32_t *lut_image;    // 128 KB table image from ep_prepare_tables / the table-build launch, or null: build the
                                  // tables here (b <= 11 only)
    const uint32_t *cold;         // b = 12: entries of all codes of the sixteen coordinate tables, and
    uint32_t hs2;                 //         twice the first code of the hot window
    uint32_t off_freq;            // byte offset of the u16 frequency arrays inside the blob
    uint32_t off_payload;
    uint32_t total_words;
    uint32_t n_vec;
    uint32_t per_row;             // C / 8
    uint32_t V, n_tiles, b;       // n_tiles: tiles of the whole tensor
    uint32_t tile0, tile_cnt;     // the tiles this launch decodes: [tile0, tile0 + tile_cnt)
    int32_t zlo;                  // even, <= -2
    uint32_t rounds;              // ceil(tile_cnt / tiles per round): in one round the warps of a CTA take consecutive tiles
    uint32_t round_cost;          // work of one round in groups of 32 vectors (ceil(V / 32)), or 1 (see split_rounds)
    uint32_t cost_begin;          // sum of rounds * round_cost over the jobs before this one
    uint32_t row_bytes;           // output bytes per row
    uint32_t row_rcp;             // ceil(2^32 / row_bytes)
    uint32_t row_max;             // index of the last row
    float payload_bits;           // mean payload bits per symbol
    uint32_t guess;               // decode_tile_few: the loop that guesses (see EP_BODY11_GUESS)
    int16_t tmin[EP_NUM_TABLES];
    uint16_t tK[EP_NUM_TABLES];
    uint16_t foff[EP_NUM_TABLES]; // start of table t's frequencies, in u16 units
};

struct BatchParams {
    JobParams job[EP_MAX_BATCH];
    uint32_t cost_per_cta;        // ceil(sum of rounds * round_cost over all jobs / CTAs of the launch)
    uint32_t tiles_per_round;     // tiles a CTA works on at a time: one per warp, at most kTilesPerRound
    int32_t n_jobs;
};

// ---- small PTX helpers -------------------------------------------------------------------------
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t addr, uint64_t v) {
    asm volatile("st.shared.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, uint64_t src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Programmatic launch: a kernel of this file may come up while the kernel before it in the stream still runs, and lets the
// next one come up likewise.  Nothing is read or written before this wait, which ends when everything earlier in the stream
// has, so the order of effects is the stream's; what overlaps is the launch itself (see launch_next).
__device__ __forceinline__ void wait_for_stream() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// two fp32 lanes per instruction (sm_100 packed fp32), operands kept as 64-bit register pairs
__device__ __forceinline__ uint64_t pack64(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ void unpack64(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// snap_tau of Eq. 19 for two neighbouring weights (lo = lower address)
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack_fp16_sat(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.satfinite.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack_e4m3(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack_e5m2(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t cvt_u8(float v) {
    uint32_t r;
    asm("cvt.rni.sat.u8.f32 %0, %1;" : "=r"(r) : "f"(v));
    return r & 0xFFu;
}
__device__ __forceinline__ uint32_t cvt_s8(float v) {
    int32_t r;
    asm("cvt.rni.sat.s8.f32 %0, %1;" : "=r"(r) : "f"(v));
    return uint32_t(r) & 0xFFu;
}

// ---- lookup-table construction (per CTA, from the stream's frequency tables) ---------------------
// Warp t - 1 fills coordinate table t (t = 1..16; the coset table t = 0 needs none).  Symbols are taken 32 at
// a time: a warp scan gives each lane its symbol's first slot, every lane writes the first sixteen slots of
// its own symbol, and the few symbols with more slots than that are then filled by the whole warp, one
// after the other (that loop is serial: its length, not the number of stores, is what the build time
// depends on).  `put` stores an entry.  (A prepared table image: ep_prepare_tables_kernel.)
template <class Store>
__device__ __forceinline__ void build_one_table(const JobParams &J, uint32_t t, uint32_t lane, Store put) {
    const uint32_t K = J.tK[t];
    const uint16_t *fq = reinterpret_cast<const uint16_t *>(J.stream + J.off_freq) + J.foff[t];
    const int32_t tmin = J.tmin[t];
    const bool is_m = ((t - 1) & 7) == 7;
    const uint32_t slots = min(1u << J.b, kLutEntries);
    uint32_t run = 0;
    for (uint32_t j0 = 0; j0 < K; j0 += 32) {
        const uint32_t j = j0 + lane;
        const uint32_t f = j < K ? uint32_t(fq[j]) : 0u;
        uint32_t incl = f;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= uint32_t(d)) incl += n;
        }
        const uint32_t first = run + incl - f;
        const int32_t v = tmin + int32_t(j);
        const uint32_t code = uint32_t((is_m ? 2 * v : v) - J.zlo);
        // (a frequency of 2^11 or more is not a stream the launcher sends here: it does not fit its field; whatever the
        // device copy holds, an entry's frequency stays in 1 .. 2047, which the word bound of the ring relies on)
        const uint32_t entry = (min(f, kLutEntries - 1u) << 21) | ((code & 0x3FFu) << 11);
        if (f >= kLutEntries) atomicOr(&g_ep_status, 1u);
#pragma unroll
        for (uint32_t u = 0; u < kOwnSlots; ++u)
            if (u < f && first + u < slots) put(first + u, entry | u);
        uint32_t big = __ballot_sync(0xFFFFFFFFu, f > kOwnSlots);
        while (big) {
            const int i = __ffs(big) - 1;
            big &= big - 1;
            const uint32_t fi = __shfl_sync(0xFFFFFFFFu, f, i);
            const uint32_t Fi = __shfl_sync(0xFFFFFFFFu, first, i);
            const uint32_t ei = __shfl_sync(0xFFFFFFFFu, entry, i);
            for (uint32_t u = kOwnSlots + lane; u < fi && Fi + u < slots; u += 32) put(Fi + u, ei | u);
        }
        run += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    // frequencies of a damaged stream may sum to less than 2^b, and a table may be empty: a slot that no symbol
    // owns gets f = 1, never what an earlier job left there (the word bound of the ring relies on f >= 1)
    for (uint32_t u = min(run, slots) + lane; u < slots; u += 32) put(u, kEntryUnused);
}

__device__ __forceinline__ void build_tables_smem(const JobParams &J, uint32_t lut_addr, uint32_t warp, uint32_t lane) {
    for (uint32_t t = 1 + warp; t < EP_NUM_TABLES; t += blockDim.x >> 5) {
        const uint32_t base = lut_addr + (t - 1) * kLutStride;
        build_one_table(J, t, lane, [base](uint32_t slot, uint32_t e) { sts32(base + 4u * slot, e); });
    }
}

// the prepared image of the same sixteen tables, 128 KB: one thread asks for it, the copy engine brings it in.  (256 threads
// with 16 bytes per cp.async kept the load pipe busy for a microsecond, and the first tile's payload queued behind
// it: 3.6 us from a launch's turn to its first group.)  Whoever reads the tables waits for the mbarrier first.
// One copy: asking for four of 32 KB took the asking warp 0.8 us, by which its own tile then began later (8192 x 8192 at 4 bpp 59.25 -> 59.0 us,
// block of seven at 2.5 bpp to FP8 302.9 -> 300.4, at 3.5 to BF16 310.5 -> 309.5).  Asked for by another warp - one more than tiles, or the
// last - the same, and 1 % slower where few tiles decode without the guess.
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void copy_tables_smem(const uint32_t *image, uint32_t lut_addr, uint32_t bar, bool two_level) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kLutBytes + (two_level ? kHotBytes : 0u)) : "memory");
    auto piece = [&](uint32_t dst, uint32_t src, uint32_t bytes) {
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(dst), "l"(reinterpret_cast<uint64_t>(image) + src), "r"(bytes), "r"(bar) : "memory");
    };
    piece(lut_addr, 0u, kLutBytes);
    if (two_level) piece(lut_addr + kHotBase, kLutBytes, kHotBytes);      // the hot part of the second level follows the image
}

// How the job's lookup tables come about, and the wait for them.  All branches are on votes or parameters (a guard around each
// vote of the hot loop costs more than the wait).  A copy that does not end within the limit - there is no such case -
// raises the integrity word and ends the warp, whose tiles are not written: what an SM's shared memory held before has neither
// frequencies of at least 1 nor codes inside the second level, which the loops' addresses rely on.  (A barrier that waits for
// all threads of a CTA does not wait for those that have ended, and only a warp that saw a phase end arms the next one.)
enum TablesPending : uint32_t { kTablesThere, kTablesBuilt, kTablesCopied };   // nothing to wait for; this CTA's stores; the copy
struct TablesWait { uint32_t pending, bar, parity; };
static_assert(EP_MAX_BATCH <= kWarps);
constexpr uint32_t kSpinLimit = 1u << 18;             // attempts of about a microsecond each at most: a quarter of a second
__device__ __forceinline__ void wait_for_tables(const TablesWait &W) {
    if (W.pending == kTablesBuilt) __syncthreads();
    if (W.pending == kTablesCopied) {
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 left;\n\tmov.b32 left, %2;\n\t"
                     "EP_TABLES_WAIT:\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1, 1000;\n\t"
                     "vote.sync.all.pred p, p, 0xffffffff;\n\t"
                     "@p bra.uni EP_TABLES_DONE;\n\t"
                     "sub.u32 left, left, 1;\n\t"
                     "setp.ne.u32 p, left, 0;\n\t"
                     "vote.sync.all.pred p, p, 0xffffffff;\n\t"
                     "@p bra.uni EP_TABLES_WAIT;\n\t"
                     "red.global.or.b32 [%3], 2;\n\t"
                     "exit;\n\t"
                     "EP_TABLES_DONE:\n\t}"
                     ::"r"(W.bar), "r"(W.parity), "n"(kSpinLimit), "l"(&g_ep_status) : "memory");
    }
}

// frequencies of the two cosets as the decode uses them: u < f0 means coset 0.  A coset that never occurs
// has frequency 0 in the stream and is never selected; it is raised to 1 here only so that a damaged stream
// cannot produce a state that takes a word in every step.
struct CosetFreq { uint32_t f0, f1; };
__device__ __forceinline__ CosetFreq load_coset(const JobParams &J) {
    const uint16_t *fq = reinterpret_cast<const uint16_t *>(J.stream + J.off_freq) + J.foff[0];
    uint32_t f0 = 0, f1 = 0;
    if (J.tmin[0] == 0) {
        f0 = __ldg(fq);
        if (J.tK[0] > 1) f1 = __ldg(fq + 1);
    } else {
        f1 = __ldg(fq);
    }
    const uint32_t M = 1u << J.b;
    CosetFreq c;
    c.f0 = min(f0, M);                 // u < f0 <=> coset 0 (f0 = 0: never)
    c.f1 = max(min(f1, M), 1u);
    return c;
}

// ---- one rANS symbol (Eq. 18) followed by renormalisation: plain version --------------------------
// x: this lane's state; wa: shared-memory byte address of the tile's word cursor (same in all lanes).
// Lanes that need a word take them in lane order: lane l reads the word popc(ballot & lanes below l)
// places after the cursor; the cursor then advances by popc(ballot) words.  Lanes without a vector
// (`act` false: the last, partly filled group of a tile) leave their state alone and take no word.
__device__ __forceinline__ void renorm_plain(uint32_t &x, uint32_t &wa, uint32_t lt, bool need) {
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, need);
    if (need) {
        uint16_t w;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(w) : "r"(wa + 2u * __popc(bal & lt)));
        x = (x << 16) | w;
    }
    wa += 2u * __popc(bal);
}
__device__ __forceinline__ uint32_t rans_step_plain(uint32_t &x, uint32_t table_addr, uint32_t mask, uint32_t b, uint32_t &wa,
                                                    uint32_t lt, bool act) {
    uint32_t e = 0;
    bool need = false;
    if (act) {
        e = lds32(table_addr + ((x & mask) << 2));
        x = (e >> 21) * (x >> b) + (e & 0x7FFu);
        need = x < ep::kStateLow;
    }
    renorm_plain(x, wa, lt, need);
    return e;
}
// the coset symbol: 0 if the slot lies below f0, else 1
__device__ __forceinline__ uint32_t coset_step_plain(uint32_t &x, CosetFreq cf, uint32_t mask, uint32_t b, uint32_t &wa,
                                                     uint32_t lt, bool act) {
    uint32_t c = 0;
    bool need = false;
    if (act) {
        const uint32_t u = x & mask;
        c = u < cf.f0 ? 0u : 1u;
        x = (c ? cf.f1 : max(cf.f0, 1u)) * (x >> b) + (c ? u - cf.f0 : u);
        need = x < ep::kStateLow;
    }
    renorm_plain(x, wa, lt, need);
    return c;
}

template <int DT>
struct Out;   // per output type: bytes per 8-weight block and the store of one block

template <>
struct Out<EP_BF16> {
    static constexpr uint32_t kBlockBytes = 16;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        uint4 q = make_uint4(pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]), pack_bf16(w[4], w[5]), pack_bf16(w[6], w[7]));
        *reinterpret_cast<uint4 *>(dst) = q;
    }
};
template <>
struct Out<EP_FP16> {
    static constexpr uint32_t kBlockBytes = 16;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        uint4 q = make_uint4(pack_fp16_sat(w[0], w[1]), pack_fp16_sat(w[2], w[3]), pack_fp16_sat(w[4], w[5]),
                             pack_fp16_sat(w[6], w[7]));
        *reinterpret_cast<uint4 *>(dst) = q;
    }
};
template <>
struct Out<EP_FP8_E4M3> {
    static constexpr uint32_t kBlockBytes = 8;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        uint2 q = make_uint2(pack_e4m3(w[0], w[1]) | (pack_e4m3(w[2], w[3]) << 16),
                             pack_e4m3(w[4], w[5]) | (pack_e4m3(w[6], w[7]) << 16));
        *reinterpret_cast<uint2 *>(dst) = q;
    }
};
template <>
struct Out<EP_INT8> {
    static constexpr uint32_t kBlockBytes = 8;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        uint2 q = make_uint2(cvt_s8(w[0]) | (cvt_s8(w[1]) << 8) | (cvt_s8(w[2]) << 16) | (cvt_s8(w[3]) << 24),
                             cvt_s8(w[4]) | (cvt_s8(w[5]) << 8) | (cvt_s8(w[6]) << 16) | (cvt_s8(w[7]) << 24));
        *reinterpret_cast<uint2 *>(dst) = q;
    }
};

template <>
struct Out<EP_FP32> {
    static constexpr uint32_t kBlockBytes = 32;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        reinterpret_cast<float4 *>(dst)[0] = make_float4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<float4 *>(dst)[1] = make_float4(w[4], w[5], w[6], w[7]);
    }
};
template <>
struct Out<EP_FP8_E5M2> {
    static constexpr uint32_t kBlockBytes = 8;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        uint2 q = make_uint2(pack_e5m2(w[0], w[1]) | (pack_e5m2(w[2], w[3]) << 16),
                             pack_e5m2(w[4], w[5]) | (pack_e5m2(w[6], w[7]) << 16));
        *reinterpret_cast<uint2 *>(dst) = q;
    }
};
template <>
struct Out<EP_UINT8> {
    static constexpr uint32_t kBlockBytes = 8;
    static __device__ __forceinline__ void store(void *dst, const float (&w)[8]) {
        uint2 q = make_uint2(cvt_u8(w[0]) | (cvt_u8(w[1]) << 8) | (cvt_u8(w[2]) << 16) | (cvt_u8(w[3]) << 24),
                             cvt_u8(w[4]) | (cvt_u8(w[5]) << 8) | (cvt_u8(w[6]) << 16) | (cvt_u8(w[7]) << 24));
        *reinterpret_cast<uint2 *>(dst) = q;
    }
};

template <int DT>
struct BlockBytes { static constexpr uint32_t value = Out<DT>::kBlockBytes; };
template <>
struct BlockBytes<EP_FIELDS_I32> { static constexpr uint32_t value = 36; };

// ---- one group of 32 vectors, plain version: nine symbols per lane, then Eq. 5 / Eq. 19 and the store ---
template <int DT>
__device__ __forceinline__ void decode_group_plain(uint32_t &x, uint32_t &wa, uint32_t lut_addr, CosetFreq cf, uint32_t mask,
                                                   uint32_t b, uint32_t lt, bool act, uint32_t k0_bits, float sigma,
                                                   int32_t zlo, void *dst) {
    uint32_t e[9];
    const uint32_t c = coset_step_plain(x, cf, mask, b, wa, lt, act);
    const uint32_t tab = lut_addr + c * kCosetStride;
#pragma unroll
    for (int k = 1; k <= 8; ++k) e[k] = rans_step_plain(x, tab + uint32_t(k - 1) * kLutStride, mask, b, wa, lt, act);
    if (!act) return;
    // parity of z1 + ... + z7 = xor of the codes' lowest bits (zlo is even); it is the lowest bit of z8
    const uint32_t par = (e[1] ^ e[2] ^ e[3] ^ e[4] ^ e[5] ^ e[6] ^ e[7]) & 0x800u;
    if constexpr (DT == EP_FIELDS_I32) {
        int32_t *f = reinterpret_cast<int32_t *>(dst);
        f[0] = int32_t(c);
#pragma unroll
        for (int k = 1; k <= 7; ++k) f[k] = int32_t((e[k] & kCodeMask) >> 11) + zlo;
        f[8] = (int32_t((e[8] & kCodeMask) >> 11) + zlo) >> 1;
    } else {
        // (entry & mask) | 0x45800000 | c << 10 is 4096 + code + c/2 as fp32 (one ulp here is 2^-11); subtracting
        // 4096 - zlo gives p = z + c/2 exactly
        const uint32_t cc = kExp4096 | (c << 10);
        const uint64_t kk = pack64(k0_bits, k0_bits);
        const uint64_t ss = pack64(__float_as_uint(sigma), __float_as_uint(sigma));
        uint32_t xb[8];
#pragma unroll
        for (int k = 1; k <= 7; ++k) xb[k - 1] = (e[k] & kCodeMask) | cc;
        xb[7] = (e[8] & kCodeMask) | par | cc;
        float w[8];
#pragma unroll
        for (int i = 0; i < 8; i += 2) unpack64(mul2(sub2(pack64(xb[i], xb[i + 1]), kk), ss), w[i], w[i + 1]);
        Out<DT>::store(dst, w);
    }
}

// ---- payload ring ------------------------------------------------------------------------------------
// chunk c of a tile = global bytes [a0 + CHUNK c, a0 + CHUNK (c + 1)), a0 = tile's first word rounded down to
// 16 bytes; it lives in ring slot c mod SLOTS, and a chunk in one of the slots that make up the ring's first 512
// bytes is written a second time behind the ring's end.  `room` = bytes from a0 to the end of the payload: nothing
// beyond it is read (cp.async zero-fills the rest).  The decode kernel's rings are 3 x 512 bytes; the kernel that
// feeds the tensor cores needs the shared memory for its operands and takes 4 x 256 where these leave no more (see GemmShape).
template <uint32_t CHUNK = kChunk, uint32_t SLOTS = kRingSlots>
__device__ __forceinline__ void ring_issue(uint32_t ring, uint64_t a0, uint32_t room, uint32_t c, uint32_t lane) {
    if (lane < CHUNK / 16u) {
        uint32_t o = CHUNK * c + 16u * lane;
        uint32_t n = 16;
        if (o + 16u > room) {
            n = o < room ? room - o : 0u;
            if (n == 0) o = 0;                   // nothing is read, but keep the address a valid one
        }
        const uint32_t slot = c % SLOTS;
        const uint32_t dst = ring + CHUNK * slot + 16u * lane;
        cp_async16(dst, a0 + o, n);
        if (slot < kRingMirror / CHUNK) cp_async16(dst + CHUNK * SLOTS, a0 + o, n);
    }
    cp_async_commit();
}

// The cursor entered a new chunk: request chunks up to SLOTS - 1 ahead of it and wait for all but the
// newest.  `threshold` = start of the chunk after the cursor's at the previous service; chunks up to
// threshold / CHUNK + SLOTS - 2 have been requested.  A group touches at most 448 + 62 bytes from its start,
// which the chunks complete after this call cover (1024 bytes from the cursor's chunk on, or 768).
template <uint32_t CHUNK = kChunk, uint32_t SLOTS = kRingSlots>
__device__ __forceinline__ void ring_service(uint32_t ring, uint64_t a0, uint32_t room, uint32_t pos, uint32_t &threshold,
                                             uint32_t lane) {
    const uint32_t cur = pos / CHUNK;
    for (uint32_t c = threshold / CHUNK + SLOTS - 1u; c < cur + SLOTS; ++c) ring_issue<CHUNK, SLOTS>(ring, a0, room, c, lane);
    cp_async_wait<1>();
    __syncwarp();
    threshold = CHUNK * (cur + 1u);
}

// what a warp needs to know about its tile
struct TileSetup {
    uint32_t x;            // this lane's state, forced into [2^15, 2^31) (a no-op for a valid stream)
    uint32_t off, end;     // first payload word of the tile and of the next one
    uint32_t v0, nv;       // first block and number of blocks
    uint64_t a0;           // global address of chunk 0
    uint32_t lead, room;   // cursor position inside chunk 0; payload bytes from a0 on
};
// from a record's words: this lane's state, the tile's and the next one's first payload word (the blocks are left to the caller)
__device__ __forceinline__ TileSetup tile_setup(const JobParams &J, uint32_t state, uint32_t off, uint32_t end) {
    TileSetup T;
    T.x = max(state & 0x7FFFFFFFu, ep::kStateLow);
    T.off = min(off, J.total_words);        // a damaged index must not move reads outside the payload
    T.end = end;
    T.v0 = T.nv = 0;
    const uint64_t pay = reinterpret_cast<uint64_t>(J.stream + J.off_payload);
    const uint64_t first = pay + 2ull * T.off;
    T.a0 = first & ~15ull;
    T.lead = uint32_t(first - T.a0);
    T.room = uint32_t(pay + 2ull * J.total_words - T.a0);     // the payload is shorter than 2 GB
    return T;
}
__device__ __forceinline__ TileSetup tile_setup(const JobParams &J, uint32_t tile, bool valid, uint32_t lane) {
    const uint32_t *rec = J.tile_index + size_t(tile) * 33u;
    TileSetup T = tile_setup(J, rec[lane], rec[32], (tile + 1 < J.n_tiles) ? rec[33 + 32] : rec[33]);
    T.v0 = tile * J.V;
    T.nv = valid ? min(J.V, J.n_vec - T.v0) : 0u;
    return T;
}

// Plain C++ version of the tile loop, used for the field-dump mode, for streams with b < 11 and for tensors with
// fewer than 32 blocks per row (a group may then cross several rows).
template <int DT>
__device__ __forceinline__ void decode_tile_plain(const JobParams &J, uint32_t tile, uint32_t lut_addr, CosetFreq cf,
                                                  uint32_t ring, uint32_t lane) {
    const TileSetup T = tile_setup(J, tile, true, lane);
    uint32_t x = T.x;
    const uint32_t b = J.b, mask = (1u << b) - 1u, lt = (1u << lane) - 1u;
    const uint32_t per_row = J.per_row;
    uint32_t pos = T.lead;        // byte position of the cursor relative to a0
    uint32_t threshold;           // next chunk boundary the cursor has not yet crossed
    for (uint32_t c = 0; c < kRingSlots; ++c) ring_issue(ring, T.a0, T.room, c, lane);
    cp_async_wait<1>();
    __syncwarp();
    threshold = kChunk;
    const uint32_t k0_bits = __float_as_uint(float(4096 - J.zlo));
    const uint32_t row_max = J.n_vec / per_row - 1u;
    for (uint32_t g = 0; g * 32u < T.nv; ++g) {
        if (pos >= threshold) ring_service(ring, T.a0, T.room, pos, threshold, lane);
        const uint32_t wa0 = ring + pos % kRingBytes;
        uint32_t wa = wa0;
        const uint32_t i = g * 32u + lane;
        const bool act = i < T.nv;
        const uint32_t v = T.v0 + i;
        const float sigma = (DT == EP_FIELDS_I32) ? 0.f : __ldg(J.scales + min(v / per_row, row_max));
        decode_group_plain<DT>(x, wa, lut_addr, cf, mask, b, lt, act, k0_bits, sigma, J.zlo,
                               static_cast<uint8_t *>(J.out) + size_t(v) * BlockBytes<DT>::value);
        pos += wa - wa0;
    }
    cp_async_wait<0>();          // nothing may still be landing in the ring when the next tile starts
    __syncwarp();
    // integrity: the encoder started every state at 2^15 and the tile's words end where the next tile's begin
    const bool bad = (x != ep::kStateLow) || (T.off + ((pos - T.lead) >> 1) != T.end);
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&g_ep_status, 1u);
}

// ---- the hot loop in PTX -------------------------------------------------------------------------------------
// All groups of a tile, written as one asm statement so that every branch can be marked warp-uniform (bra.uni) and the rare
// work - refilling the payload ring, moving to the next row, the tile's end - sits out of line behind ONE warp vote per loop
// pass.
//
// Word addresses.  Lane l keeps its own address a_l of the word it would take in the current step.
// With bal_k the ballot of the lanes that need a word after step k,
//     a_l(k) = a_l(k-1) + 2 popc((bal_k & below_l) | (bal_{k-1} & ~below_l)):
// the words taken in step k-1 by lanes l and above, plus those taken in step k by the lanes below.  The two
// masks are disjoint, so one bit-select and ONE population count per step replace the prefix count and the
// cursor advance (lane 0's address is the tile's word cursor before the step).
//
// Loop-carried: x state, a word address, bal last ballot, doff byte offset of this lane's block in the
// output; inside the asm: lim = first doff at which this lane leaves its row or the tile, wthr = ring address at
// which the cursor leaves its 512-byte chunk (minus 2), ss = the row scale twice, act = lane has a block.
// A warp without a tile runs with all lanes inactive: states and addresses stand still, nothing is stored.
//
// asm operands: x, a, bal, doff are %0 .. %3; then come the inputs, named here:
#define EP_LT "%4"      /* lanes below this one (mask) */
#define EP_LUT0 "%5"    /* tables of coset 0 */
#define EP_LUT1 "%6"    /* tables of coset 1 */
#define EP_CTX "%7"     /* this warp's context block */
#define EP_KK "%8"      /* {4096 - zlo, 4096 - zlo} as fp32 pair */
#define EP_OUT "%9"     /* output base address */
#define EP_F0 "%10"     /* frequency of coset 0 */
#define EP_F1 "%11"     /* frequency of coset 1, at least 1 */
#define EP_L16 "%12"    /* 16 * lane */
#define EP_L2B "%13"    /* 2^12-slot streams: the complete second-level array (global memory), */
#define EP_HS2 "%14"    /* twice the first code of the hot window, */
#define EP_HOTOFF "%15" /* offset of the hot part in shared memory */

#define EP_CM "0x1FF800"
// One macro per line of the loop body.  E = name of the entry register (a suffix is added), OFF = byte offset of the field's table,
// BIN / BOUT = the register that holds the previous / receives the new ballot.
// a coordinate field: table OFF / 8192 of the lane's coset (Eq. 18)
// slot address 4 (x & 0x7FF) + tab as 4 x - 8192 (x >> 11) + tab: two multiply-adds instead of a mask and one (the
// multiply-add pipe has room, the ALU pipe has not; measured + 0.3 % / + 0.8 % on the 8192^2 tensor / the layer).  4 x + tab
// comes first: it is there when the shift is, so the lookup waits for one multiply-add behind the shift, not for two.  The warps
// of a full SM spend 62 % of their cycles waiting for operands, so four cycles per step are felt: 8192 x 8192 at 4 bpp to FP16 59.76 ->
// 59.2 us, block of seven at 3.5 bpp to BF16 313.7 -> 310.6, at 2.5 bpp to FP8 303.6 -> 302.9 (streams of 2^12 slots have lookups of their own).
#define EP_L1 "mad.lo.u32 uA, %0, 4, tabA;\n\t" "shr.u32 qA, %0, 11;\n\t"
#define EP_L2 "mad.lo.u32 uA, qA, 0xFFFFE000, uA;\n\t"
#define EP_L3(E, OFF) "ld.shared.u32 " E "A, [uA+" OFF "];\n\t"
#define EP_L5(E) "shr.u32 fA, " E "A, 21;\n\t"
#define EP_L6(E) "and.b32 biA, " E "A, 0x7FF;\n\t"
#define EP_L7 "@actA mad.lo.u32 %0, fA, qA, biA;\n\t"
// renormalisation: lanes whose state fell below 2^15 take a word each, in lane order
#define EP_L8 "setp.lt.and.u32 pA, %0, 32768, actA;\n\t"
#define EP_L9(BOUT) "vote.sync.ballot.b32 " BOUT ", pA, 0xffffffff;\n\t"
#define EP_L10(BIN, BOUT) "lop3.b32 tA, " EP_LT ", " BOUT ", " BIN ", 0xCA;\n\t"
#define EP_L11 "popc.b32 tA, tA;\n\t"
#define EP_L12 "mad.lo.u32 %1, tA, 2, %1;\n\t"
#define EP_L13 "ld.shared.u16 wA, [%1];\n\t"
#define EP_L14 "@pA mad.lo.u32 %0, %0, 65536, wA;\n\t"
#define EP_RENORM_ALL(BIN, BOUT) EP_L8 EP_L9(BOUT) EP_L10(BIN, BOUT) EP_L11 EP_L12 EP_L13 EP_L14
#define EP_STEP_ALL(E, OFF, BIN, BOUT) EP_L1 EP_L2 EP_L3(E, OFF) EP_L5(E) EP_L6(E) EP_L7 EP_RENORM_ALL(BIN, BOUT)
// the coset: slot below f0 -> coset 0 with frequency f0 (then at least 1), else coset 1 with frequency f1 and offset f0
#define EP_C1 "and.b32 uA, %0, 0x7FF;\n\t"
#define EP_C2 "shr.u32 qA, %0, 11;\n\t"
#define EP_C3 "setp.lt.u32 pcA, uA, " EP_F0 ";\n\t"
#define EP_C4 "selp.b32 fA, " EP_F0 ", " EP_F1 ", pcA;\n\t"
#define EP_C5 "@!pcA sub.u32 uA, uA, " EP_F0 ";\n\t"
#define EP_C6 "@actA mad.lo.u32 %0, fA, qA, uA;\n\t"
#define EP_C7 "selp.b32 tabA, " EP_LUT0 ", " EP_LUT1 ", pcA;\n\t"
#define EP_C8 "selp.b32 ccA, c0r, c1r, pcA;\n\t"
#define EP_COSET_ALL                                                                                 \
    EP_C1 EP_C2 EP_C3 EP_C4 EP_C5 EP_C6 EP_C7 EP_C8                                                                   \
    EP_RENORM_ALL("%2", "naA")
// Eq. 5 and the product of Eq. 19 for two neighbouring weights: 4096 + code (+ 1/2) as fp32, minus 4096 - zlo, times sigma
#define EP_XA(E) "lop3.b32 xaA, " E "A, " EP_CM ", ccA, 0xEA;\n\t"
#define EP_XB(E) "lop3.b32 xbA, " E "A, " EP_CM ", ccA, 0xEA;\n\t"
#define EP_P1 "mov.b64 prA, {xaA, xbA};\n\t"
#define EP_P2 "sub.rn.f32x2 prA, prA, " EP_KK ";\n\t"
#define EP_P3 "mul.rn.f32x2 prA, prA, ssA;\n\t"
#define EP_P4 "mov.b64 {wlA, whA}, prA;\n\t"
#define EP_PAIR_ALL EP_P1 EP_P2 EP_P3 EP_P4
// parity of z1 + ... + z7 = xor of the codes' lowest bits (bit 11 of the entries; zlo is even): the lowest bit of z8
#define EP_PAR3(EA, EB, EC) "lop3.b32 parA, " EA "A, " EB "A, " EC "A, 0x96;\n\t"
#define EP_PARX "lop3.b32 parA, parA, 0x800, ccA, 0xEA;\n\t"
#define EP_X8 "lop3.b32 xbA, e8A, " EP_CM ", parA, 0xEA;\n\t"
#define EP_ADDR "mad.wide.u32 adA, %3, 1, " EP_OUT ";\n\t"

// ---- streams with 2^12 slots per table (b = 12: the paper's setting for 8 bpp targets) ------------------------
// Sixteen tables of 4096 four-byte entries would not fit shared memory, so the lookup has two levels.  Shared memory
// holds, per slot, 16 bits: twice the code of the slot's coordinate value, code = z - zlo (2m - zlo for the m field;
// the same 128 KB and strides as the one-level tables of b = 11).  The code is all Eq. 5 needs - it goes into the
// mantissa of 2^22 (bit 0 = the coset's half, bit 1 = one) - and it addresses the second level, one word per (table,
// code): f << 16 | F.  Entries of the kHotSpan codes around zero sit in shared memory, all of them in global memory.
// HOFF / COFF = byte offset of the field's table in the hot part / in the complete array.
#define EP_N1 "and.b32 uA, %0, 0xFFF;\n\t"
#define EP_N2 "mad.lo.u32 tA, uA, 2, tabA;\n\t"
#define EP_N3(E, OFF) "ld.shared.u16 " E "A, [tA+" OFF "];\n\t"
/* codes inside the hot window: entry in shared memory; the others: global memory */
#define EP_N4(E) "sub.u32 wA, " E "A, " EP_HS2 ";\n\t"
#define EP_N5 "setp.lt.u32 pcA, wA, 1056;\n\t"
#define EP_N6 "mad.lo.u32 tA, wA, 2, hotcA;\n\t"
#define EP_N7(E) "mad.wide.u32 adA, " E "A, 2, lcA;\n\t"
#define EP_N8(HOFF, COFF)                                                                                             \
    "@pcA ld.shared.u32 wA, [tA+" HOFF "];\n\t" "@!pcA ld.global.nc.u32 wA, [adA+" COFF "];\n\t"
#define EP_N9 "shr.u32 qA, %0, 12;\n\t"
#define EP_N10 "shr.u32 fA, wA, 16;\n\t"
#define EP_N11 "and.b32 biA, wA, 0xFFFF;\n\t"
#define EP_N12 "sub.u32 biA, uA, biA;\n\t"
#define EP_N13 "@actA mad.lo.u32 %0, fA, qA, biA;\n\t"
#define EP_STEP12_ALL(E, OFF, BIN, BOUT, HOFF, COFF)                                                                  \
    EP_N1 EP_N2 EP_N3(E, OFF) EP_N4(E) EP_N5 EP_N6 EP_N7(E) EP_N8(HOFF, COFF) EP_N9 EP_N10 EP_N11 EP_N12 EP_N13 EP_RENORM_ALL(BIN, BOUT)
#define EP_C1_12 "and.b32 uA, %0, 0xFFF;\n\t"
#define EP_C2_12 "shr.u32 qA, %0, 12;\n\t"
/* per coset: 2^22 (+ 1/2) as fp32, the hot part and the complete array of its eight tables */
#define EP_C8_12 "selp.b32 ccA, d0r, d1r, pcA;\n\t"
#define EP_C9_12 "selp.b32 hotcA, hotb, hotb1, pcA;\n\t"
#define EP_C10_12 "selp.b64 lcA, " EP_L2B ", l2b1, pcA;\n\t"
#define EP_COSET12_ALL                                                                               \
    EP_C1_12 EP_C2_12 EP_C3 EP_C4 EP_C5 EP_C6 EP_C7                                                                   \
    EP_C8_12 EP_C9_12 EP_C10_12 EP_RENORM_ALL("%2", "naA")
// Eq. 5: 2^22 + code (+ 1/2) as fp32; z8 = 2m + parity of (z1 + ... + z7), the parity from bit 1 of the xor of the
// looked-up values (zlo is even)
#define EP_XA12(E) "or.b32 xaA, " E "A, ccA;\n\t"
#define EP_XB12(E) "or.b32 xbA, " E "A, ccA;\n\t"
#define EP_PARX12 "lop3.b32 parA, parA, 0x2, ccA, 0xEA;\n\t"
#define EP_X8_12 "or.b32 xbA, e8A, parA;\n\t"
// the nine steps and the arithmetic of one group, 2^11-slot and 2^12-slot streams
#define EP_BODY11(CVT)                                                                                                \
        EP_COSET_ALL                                                                                                  \
        EP_STEP_ALL("e1", "0", "naA", "nbA")     EP_XA("e1")                                                          \
        EP_STEP_ALL("e2", "8192", "nbA", "naA")  EP_XB("e2") EP_PAIR_ALL CVT("0")                                     \
        EP_STEP_ALL("e3", "16384", "naA", "nbA") EP_PAR3("e1", "e2", "e3") EP_XA("e3")                                \
        EP_STEP_ALL("e4", "24576", "nbA", "naA") EP_XB("e4") EP_PAIR_ALL CVT("1")                                     \
        EP_STEP_ALL("e5", "32768", "naA", "nbA") EP_PAR3("par", "e4", "e5") EP_XA("e5")                               \
        EP_STEP_ALL("e6", "40960", "nbA", "naA") EP_XB("e6") EP_PAIR_ALL CVT("2")                                     \
        EP_STEP_ALL("e7", "49152", "naA", "nbA") EP_PAR3("par", "e6", "e7") EP_XA("e7")                               \
        EP_STEP_ALL("e8", "57344", "nbA", "%2") EP_PARX EP_X8 EP_PAIR_ALL CVT("3")
#define EP_BODY12(CVT)                                                                                                \
        EP_COSET12_ALL                                                                                                \
        EP_STEP12_ALL("e1", "0", "naA", "nbA", "0", "0")             EP_XA12("e1")                                    \
        EP_STEP12_ALL("e2", "8192", "nbA", "naA", "2112", "16384")   EP_XB12("e2") EP_PAIR_ALL CVT("0")               \
        EP_STEP12_ALL("e3", "16384", "naA", "nbA", "4224", "32768")  EP_PAR3("e1", "e2", "e3") EP_XA12("e3")          \
        EP_STEP12_ALL("e4", "24576", "nbA", "naA", "6336", "49152")  EP_XB12("e4") EP_PAIR_ALL CVT("1")               \
        EP_STEP12_ALL("e5", "32768", "naA", "nbA", "8448", "65536")  EP_PAR3("par", "e4", "e5") EP_XA12("e5")         \
        EP_STEP12_ALL("e6", "40960", "nbA", "naA", "10560", "81920") EP_XB12("e6") EP_PAIR_ALL CVT("2")               \
        EP_STEP12_ALL("e7", "49152", "naA", "nbA", "12672", "98304") EP_PAR3("par", "e6", "e7") EP_XA12("e7")         \
        EP_STEP12_ALL("e8", "57344", "nbA", "%2", "14784", "114688") EP_PARX12 EP_X8_12 EP_PAIR_ALL CVT("3")

// ---- the same group with a shorter chain, for few tiles per SM (2^11-slot streams) ---------------------------------
// With a couple of warps per scheduler the time of a group is the latency of its nine steps, and in EP_BODY11 a step is one
// chain: slot address and lookup (41 cycles), new state (8), ballot (18), rank (20), word (29), back into the state (4).
// EP_BODY11_SHORT: the next slot is taken from the word itself, not from the state that the word goes into (va = the word
// where one was taken, else the state: their low eleven bits are the same).  1362 -> 1276 cycles per group (one tile per SM, 2.5 bpp to
// BF16, launches of 1792- and 3640-block tiles compared, 1965 MHz).
#define EP_T_RENORM(BIN, BOUT)                                                                                        \
        "setp.lt.and.u32 pA, %0, 32768, actA;\n\t" "vote.sync.ballot.b32 " BOUT ", pA, 0xffffffff;\n\t"               \
        "mov.b32 va, %0;\n\t" "lop3.b32 tA, " EP_LT ", " BOUT ", " BIN ", 0xCA;\n\t" "popc.b32 tA, tA;\n\t"           \
        "mad.lo.u32 %1, tA, 2, %1;\n\t" "@pA ld.shared.u16 va, [%1];\n\t"
#define EP_T_TAKE "@pA mad.lo.u32 %0, %0, 65536, va;\n\t"
#define EP_T_STEP(E, OFF, BIN, BOUT)                                                                                  \
        "and.b32 uA, va, 0x7FF;\n\t" "mad.lo.u32 uA, uA, 4, tabA;\n\t" "ld.shared.u32 " E "A, [uA+" OFF "];\n\t"      \
        "shr.u32 qA, %0, 11;\n\t" "shr.u32 fA, " E "A, 21;\n\t" "and.b32 biA, " E "A, 0x7FF;\n\t"                     \
        "@actA mad.lo.u32 %0, fA, qA, biA;\n\t" EP_T_RENORM(BIN, BOUT) EP_T_TAKE
#define EP_T_COSET                                                                                                    \
        EP_C1 EP_C2 EP_C3 EP_C4 EP_C5 EP_C6 EP_C7 EP_C8
#define EP_BODY11_SHORT(CVT)                                                                                          \
        EP_T_COSET EP_T_RENORM("%2", "naA") EP_T_TAKE                                                                 \
        EP_T_STEP("e1", "0", "naA", "nbA")     EP_XA("e1")                                                            \
        EP_T_STEP("e2", "8192", "nbA", "naA")  EP_XB("e2") EP_PAIR_ALL CVT("0")                                       \
        EP_T_STEP("e3", "16384", "naA", "nbA") EP_PAR3("e1", "e2", "e3") EP_XA("e3")                                  \
        EP_T_STEP("e4", "24576", "nbA", "naA") EP_XB("e4") EP_PAIR_ALL CVT("1")                                       \
        EP_T_STEP("e5", "32768", "naA", "nbA") EP_PAR3("par", "e4", "e5") EP_XA("e5")                                 \
        EP_T_STEP("e6", "40960", "nbA", "naA") EP_XB("e6") EP_PAIR_ALL CVT("2")                                       \
        EP_T_STEP("e7", "49152", "naA", "nbA") EP_PAR3("par", "e6", "e7") EP_XA("e7")                                 \
        "and.b32 uA, va, 0x7FF;\n\t" "mad.lo.u32 uA, uA, 4, tabA;\n\t" "ld.shared.u32 e8A, [uA+57344];\n\t"           \
        "shr.u32 qA, %0, 11;\n\t" "shr.u32 fA, e8A, 21;\n\t" "and.b32 biA, e8A, 0x7FF;\n\t"                           \
        "@actA mad.lo.u32 %0, fA, qA, biA;\n\t" EP_T_RENORM("nbA", "%2")                                              \
        EP_PARX EP_X8 EP_PAIR_ALL CVT("3")
#define EP_SHORT_FIN EP_T_TAKE      /* the last words go into the states after the loop's test: its vote fills the wait */

// EP_BODY11_GUESS: a lane that takes a word in step k hardly ever takes another in step k + 1 (its state is then at least
// 2^20 and usually above 2^26, and a step shortens a state by eleven bits at most), and no other lane needs a word to go on.
// So the ballot of step k + 1 is taken of the lanes that did not take a word in step k, whose lookup has not waited for
// step k's words.  The lanes that did follow with a lookup of their own and are back for the lookup of step k + 2.  If one
// of them falls below 2^15 all the same (`lm`, the smallest such state), the ballots were wrong, and the group is decoded
// again from its saved start by EP_BODY11_SHORT: no result depends on the guess.
// The body is for groups in which every lane has a block (a tile's last one, if it is not full, takes EP_BODY11_SHORT), so its updates
// carry no lane's flag: 25 instructions per step with the two fences, 27 with flags (EP_T_STEP has 15).
// The order below follows the times at which operands arrive (a warp issues in order): rank of the words, the late lanes'
// end of the previous step (TAIL, predicate NP from two steps ago), lookup, word, work for the output (FILL), new state, the late
// lanes' lookup, ballot.  Kept, it is 750 cycles per group by the latencies of the instructions (logic and multiply-add 4, population
// count 17, comparison and ballot 17, shared memory 25).  The assembler has an order of its own, and moves nothing across a
// signal to dependent launches, which has no effect after the kernel's first one and takes 4 cycles, nor across a read of
// the clock, which takes 10 (and whose value has to be used: KEEP, once per tile): one after the word's load and one after the
// ballot or at the step's end keep the order.  (That is a property of this assembler, CUDA 12.9, not of the language: another one is
// warned of below.)  Which is best
// depends on what the output takes.  1792-block tiles at 3.5 bpp, us, three / eight tiles per SM, signals at the end, signals after
// the ballot, clock reads after the ballot: BF16 32.7 / 36.0, 33.1 / 36.5, 33.2 / 36.7 (without fences, never-taken branches or warp
// barriers 36 and more); FP32 33.5 / 37.0, 33.0 / 36.8, 33.4 / 37.5; E4M3 33.5 / 36.9, 33.6 / 36.7, 32.8 / 36.0; INT8 33.7 / 37.0,
// 33.2 / 36.3, 32.9 / 36.6.  With the lane's flag and clock reads they took 33.4 / 37.3 (BF16), 34.3 / 38.5, 33.2 / 37.1, 33.4 / 37.6;
// EP_BODY11_SHORT takes 37.0 / 38.8.
// PB / PPB: ballots of the previous step and the one before; PP: the lanes that took a word; NB / NP: this step's.
// K: EP_K16, EP_K32 or EP_K8, by the bits of the output type
#if __CUDACC_VER_MAJOR__ != 12 || __CUDACC_VER_MINOR__ != 9
#warning "the order of EP_BODY11_GUESS was measured with CUDA 12.9: time it again, against EP_BODY11_SHORT and with other fences"
#endif
#define EP_G_SIGNAL "griddepcontrol.launch_dependents;\n\t"
#define EP_K16_WORD(E) EP_G_SIGNAL
#define EP_K16_BALLOT(E)
#define EP_K16_END EP_G_SIGNAL
#define EP_K32_WORD(E) EP_G_SIGNAL
#define EP_K32_BALLOT(E) EP_G_SIGNAL
#define EP_K32_END
#define EP_K8_WORD(E) "mov.u32 k" E ", %%clock;\n\t"
#define EP_K8_BALLOT(E) "mov.u32 l" E ", %%clock;\n\t"
#define EP_K8_END
#define EP_K8_REG(R) ".reg .b32 " R ";\n\t" "mov.b32 " R ", 0;\n\t"
#define EP_K8_ST(R) "st.volatile.shared.u32 [" EP_CTX "+60], " R ";\n\t"
#define EP_K8_ALL(DO) DO("ke1") DO("ke2") DO("ke3") DO("ke4") DO("ke5") DO("ke6") DO("ke7") DO("ke8") DO("le1") DO("le2") DO("le3") DO("le4") DO("le5") \
        DO("le6") DO("le7") DO("le8")
#define EP_K8_REGS EP_K8_ALL(EP_K8_REG)      /* (without the first values E4M3 takes 33.6 and 36.9 us instead of 32.8 and 36.0) */
#define EP_K8_KEEP EP_K8_ALL(EP_K8_ST)
#define EP_G_TAIL(P) "shr.u32 f2, ea, 21;\n\t" "and.b32 b2, ea, 0x7FF;\n\t" "@" P " mad.lo.u32 %0, f2, q2, b2;\n\t"
#define EP_G_REST(E, P) "@" P " min.u32 lm, lm, %0;\n\t" "@" P " mov.b32 " E "A, ea;\n\t"
#define EP_G_RANK(PB, PPB) "lop3.b32 tA, " EP_LT ", " PB ", " PPB ", 0xCA;\n\t" "popc.b32 tA, tA;\n\t"
#define EP_G_STEP(K, E, OFF, PB, PPB, PP, NB, NP, TAIL, REST, FILL)                                                   \
        EP_G_RANK(PB, PPB) TAIL                                                                                       \
        "and.b32 uA, %0, 0x7FF;\n\t" "mad.lo.u32 uA, uA, 4, tabA;\n\t" "ld.shared.u32 " E "A, [uA+" OFF "];\n\t"      \
        "mad.lo.u32 %1, tA, 2, %1;\n\t" "@" PP " ld.shared.u16 wA, [%1];\n\t" K##_WORD(E)                             \
        "shr.u32 qA, %0, 11;\n\t" REST FILL                                                                           \
        "shr.u32 fA, " E "A, 21;\n\t" "and.b32 biA, " E "A, 0x7FF;\n\t" "and.b32 va, wA, 0x7FF;\n\t"                  \
        "@!" PP " mad.lo.u32 %0, fA, qA, biA;\n\t" "mad.lo.u32 va, va, 4, tabA;\n\t"                                  \
        "setp.lt.and.u32 " NP ", %0, 32768, !" PP ";\n\t" "@" PP " ld.shared.u32 ea, [va+" OFF "];\n\t"               \
        "vote.sync.ballot.b32 " NB ", " NP ", 0xffffffff;\n\t" K##_BALLOT(E)                                         \
        "@" PP " mad.lo.u32 %0, %0, 65536, wA;\n\t" "shr.u32 q2, %0, 11;\n\t" K##_END
#define EP_BODY11_GUESS(K, CVT)                                                                                       \
        "mov.b32 lm, 0xffffffff;\n\t" "mov.b32 sx, %0;\n\t" "mov.b32 sa, %1;\n\t" "mov.b32 sb, %2;\n\t"               \
        EP_C1 EP_C2 EP_C3 EP_C4 EP_C5 "mad.lo.u32 %0, fA, qA, uA;\n\t" EP_C7 EP_C8                                    \
        "setp.lt.u32 pA, %0, 32768;\n\t" "vote.sync.ballot.b32 naA, pA, 0xffffffff;\n\t"                              \
        EP_G_STEP(K, "e1", "0", "naA", "%2", "pA", "nbA", "ps", "", "", "")                                              \
        EP_G_STEP(K, "e2", "8192", "nbA", "naA", "ps", "%2", "pA", EP_G_TAIL("pA"), EP_G_REST("e1", "pA"), EP_XA("e1"))  \
        EP_G_STEP(K, "e3", "16384", "%2", "nbA", "pA", "naA", "ps", EP_G_TAIL("ps"), EP_G_REST("e2", "ps"),              \
                  EP_XB("e2") EP_PAIR_ALL CVT("0"))                                                                   \
        EP_G_STEP(K, "e4", "24576", "naA", "%2", "ps", "nbA", "pA", EP_G_TAIL("pA"), EP_G_REST("e3", "pA"),              \
                  EP_PAR3("e1", "e2", "e3") EP_XA("e3"))                                                              \
        EP_G_STEP(K, "e5", "32768", "nbA", "naA", "pA", "%2", "ps", EP_G_TAIL("ps"), EP_G_REST("e4", "ps"),              \
                  EP_XB("e4") EP_PAIR_ALL CVT("1"))                                                                   \
        EP_G_STEP(K, "e6", "40960", "%2", "nbA", "ps", "naA", "pA", EP_G_TAIL("pA"), EP_G_REST("e5", "pA"),              \
                  EP_PAR3("par", "e4", "e5") EP_XA("e5"))                                                             \
        EP_G_STEP(K, "e7", "49152", "naA", "%2", "pA", "nbA", "ps", EP_G_TAIL("ps"), EP_G_REST("e6", "ps"),              \
                  EP_XB("e6") EP_PAIR_ALL CVT("2"))                                                                   \
        EP_G_STEP(K, "e8", "57344", "nbA", "naA", "ps", "%2", "pA", EP_G_TAIL("pA"), EP_G_REST("e7", "pA"),              \
                  EP_PAR3("par", "e6", "e7") EP_XA("e7"))                                                             \
        EP_G_RANK("%2", "nbA") EP_G_TAIL("ps")                                                                        \
        "mad.lo.u32 %1, tA, 2, %1;\n\t" "@pA ld.shared.u16 wA, [%1];\n\t" EP_G_REST("e8", "ps")                       \
        EP_PARX EP_X8 EP_PAIR_ALL CVT("3")
#define EP_BODY11_GUESS16(CVT) EP_BODY11_GUESS(EP_K16, CVT)
#define EP_BODY11_GUESS32(CVT) EP_BODY11_GUESS(EP_K32, CVT)
#define EP_BODY11_GUESS8(CVT) EP_BODY11_GUESS(EP_K8, CVT)
#define EP_GUESS_FIN "@pA mad.lo.u32 %0, %0, 65536, wA;\n\t"
#define EP_GUESS_INIT "mov.b32 wA, 0;\n\t" "mov.b32 ea, 0x200000;\n\t" "mov.b32 q2, 0;\n\t"

// per output type: CVT(j) turns weights 2j, 2j+1 into their stored form, STORE writes the block
#define EP_CVT_BF16(J) "cvt.rn.bf16x2.f32 o" J "A, whA, wlA;\n\t"
#define EP_CVT_FP16(J) "cvt.rn.satfinite.f16x2.f32 o" J "A, whA, wlA;\n\t"
#define EP_ST_16 "@actA st.global.v4.b32 [adA], {o0A, o1A, o2A, o3A};\n\t"
#define EP_CVT_E4M3(J) "cvt.rn.satfinite.e4m3x2.f32 h" J "A, whA, wlA;\n\t"
#define EP_CVT_E5M2(J) "cvt.rn.satfinite.e5m2x2.f32 h" J "A, whA, wlA;\n\t"
#define EP_ST_F8                                                                                                      \
    "mov.b32 o0A, {h0A, h1A};\n\t"                                                                                    \
    "mov.b32 o1A, {h2A, h3A};\n\t"                                                                                    \
    "@actA st.global.v2.b32 [adA], {o0A, o1A};\n\t"
#define EP_CVT_FP32(J) "mov.b32 ia" J "A, wlA;\n\t" "mov.b32 ib" J "A, whA;\n\t"
#define EP_ST_FP32                                                                                                    \
    "@actA st.global.v4.b32 [adA], {ia0A, ib0A, ia1A, ib1A};\n\t"                                                     \
    "@actA st.global.v4.b32 [adA+16], {ia2A, ib2A, ia3A, ib3A};\n\t"
/* one-byte integers: round to nearest even into s32 (out-of-range values end at INT_MIN / INT_MAX, NaN at 0), then
   saturate and pack four at a time: cvt.pack d, a, b, c gives (c << 16) | sat(a) << 8 | sat(b) */
#define EP_CVT_I8(J) "cvt.rni.s32.f32 ia" J "A, wlA;\n\t" "cvt.rni.s32.f32 ib" J "A, whA;\n\t"
#define EP_ST_INT8                                                                                                    \
    "cvt.pack.sat.s8.s32.b32 o2A, ib1A, ia1A, 0;\n\t"                                                                 \
    "cvt.pack.sat.s8.s32.b32 o0A, ib0A, ia0A, o2A;\n\t"                                                               \
    "cvt.pack.sat.s8.s32.b32 o3A, ib3A, ia3A, 0;\n\t"                                                                 \
    "cvt.pack.sat.s8.s32.b32 o1A, ib2A, ia2A, o3A;\n\t"                                                               \
    "@actA st.global.v2.b32 [adA], {o0A, o1A};\n\t"
#define EP_ST_UINT8                                                                                                   \
    "cvt.pack.sat.u8.s32.b32 o2A, ib1A, ia1A, 0;\n\t"                                                                 \
    "cvt.pack.sat.u8.s32.b32 o0A, ib0A, ia0A, o2A;\n\t"                                                               \
    "cvt.pack.sat.u8.s32.b32 o3A, ib3A, ia3A, 0;\n\t"                                                                 \
    "cvt.pack.sat.u8.s32.b32 o1A, ib2A, ia2A, o3A;\n\t"                                                               \
    "@actA st.global.v2.b32 [adA], {o0A, o1A};\n\t"

#define EP_REGS                                                                                                       \
    ".reg .pred pA, pcA, actA;\n\t"                                                                                   \
    ".reg .b32 uA, qA, fA, biA, tA, wA, tabA, ccA, parA, naA, nbA;\n\t"                                               \
    ".reg .b32 e1A, e2A, e3A, e4A, e5A, e6A, e7A, e8A, xaA, xbA;\n\t"                                                 \
    ".reg .b32 o0A, o1A, o2A, o3A, ia0A, ib0A, ia1A, ib1A, ia2A, ib2A, ia3A, ib3A;\n\t"                               \
    ".reg .b16 h0A, h1A, h2A, h3A;\n\t"                                                                               \
    ".reg .f32 wlA, whA, sgA;\n\t"                                                                                    \
    ".reg .b32 limA, wthrA, hotcA;\n\t"                                                                               \
    ".reg .b64 prA, ssA, adA, lcA;\n\t"
// before the first pass: the cursor leaves its first chunk at ring + chunk size - 2; lim = 0 sends the tile through EP_ROWS
#define EP_INIT                                                                                                       \
    "ld.shared.u32 r0, [" EP_CTX "+32+16];\n\t"                                                                       \
    "add.u32 wthrA, r0, 510;\n\t"                                                                                     \
    "mov.u32 limA, 0;\n\t"

#define EP_ADVANCE(GROUP_BYTES) "add.u32 %3, %3, " GROUP_BYTES ";\n\t"
// go on only if no lane left its chunk or reached its lim
#define EP_CALM_ALL "setp.lt.u32 pq, %1, wthrA;\n\t" "setp.lt.and.u32 pq, %3, limA, pq;\n\t"

// some lane reached its lim (also run once on entry): where is each lane now?
// row = doff / bytes per row by a multiply-high with ceil(2^32 / bytes per row), which is at most one too large.
#define EP_ROWS                                                                                                       \
    "setp.ge.u32 pr, %3, limA;\n\t"                                                                                   \
    "vote.sync.any.pred pr, pr, 0xffffffff;\n\t"                                                               \
    "@!pr bra.uni EP_ROWS_END_A;\n\t"                                                                                 \
    "ld.shared.v2.u32 {r0, r1}, [" EP_CTX "+8];\n\t"    /* bytes per row, last row */                          \
    "ld.shared.u32 r2, [" EP_CTX "+32+24];\n\t"     /* offset after the tile's last block */                          \
    "ld.shared.u32 r5, [" EP_CTX "+24];\n\t"                                                                   \
    "mul.hi.u32 r3, %3, r5;\n\t"                                                                                      \
    "mul.lo.u32 r4, r3, r0;\n\t"                                                                               \
    "setp.gt.u32 pv, r4, %3;\n\t"                                                                                     \
    "@pv sub.u32 r3, r3, 1;\n\t"                                                                               \
    "mad.lo.u32 r4, r3, r0, r0;\n\t"                    /* offset at which this lane enters the next row */    \
    "min.u32 limA, r4, r2;\n\t"                                                                                       \
    "setp.lt.u32 actA, %3, r2;\n\t"                                                                                   \
    "@!actA mov.u32 limA, 0xffffffff;\n\t"      /* a lane without a block never asks again */                         \
    "min.u32 r3, r3, r1;\n\t"                                                                                  \
    "ld.shared.u64 ra, [" EP_CTX "];\n\t"                                                                      \
    "mul.wide.u32 rb, r3, 4;\n\t"                                                                              \
    "add.s64 ra, ra, rb;\n\t"                                                                                  \
    "ld.global.nc.b32 r4, [ra];\n\t"                                                                           \
    "mov.b64 ssA, {r4, r4};\n\t"                                                                                      \
    "mov.b32 sgA, r4;\n\t"                                                                                            \
    "EP_ROWS_END_A:\n\t"
#define EP_ANY_ACT "or.pred pr, pr, actA;\n\t"

// The cursor left its 512-byte chunk (a group takes at most 448 + 62 bytes, so it is in the next one):
// request the chunk two ahead of the cursor's new one into the slot that became free, wait for all requests but
// this newest one, and move every address back by the ring's length when the cursor's chunk is the one in slot 0
// again.  The context keeps the request state ready to use: source address, bytes left, destination.
#define EP_SERVICE                                                                                                    \
    "setp.ge.u32 pr, %1, wthrA;\n\t"                                                                                  \
    "vote.sync.any.pred pr, pr, 0xffffffff;\n\t"                                                               \
    "@!pr bra.uni EP_SVC_END_A;\n\t"                                                                                  \
    "shfl.sync.idx.b32 r6, %1, 0, 31, 0xffffffff;\n\t"                                                                \
    "popc.b32 r0, %2;\n\t"                                                                                            \
    "mad.lo.u32 r6, r0, 2, r6;\n\t"                     /* the cursor's address */                             \
    "add.u32 r0, wthrA, 2;\n\t"                     /* end of the chunk it was in */                                  \
    "setp.lt.u32 pq, r6, r0;\n\t"                                                                              \
    "@pq bra.uni EP_SVC_END_A;\n\t"                 /* (a lane address ran ahead of the cursor: not yet) */           \
    "ld.shared.v4.u32 {r11, r12, r1, r2}, [" EP_CTX "+32];\n\t"  /* source, bytes left, destination */                \
    "ld.shared.u32 r10, [" EP_CTX "+32+16];\n\t"    /* ring base */                                                   \
    "mov.b64 ra, {r11, r12};\n\t"                                                                              \
    "sub.s32 r3, r1, " EP_L16 ";\n\t"                                                                          \
    "min.s32 r3, r3, 16;\n\t"                           /* bytes of this lane's 16 inside the payload */       \
    "setp.gt.s32 pv, r3, 0;\n\t"                        /* none: no request (nothing valid reads them) */      \
    "mad.wide.u32 rb, " EP_L16 ", 1, ra;\n\t"                                                                  \
    "add.u32 r5, r2, " EP_L16 ";\n\t"                                                                          \
    "@pv cp.async.cg.shared.global [r5], [rb], 16, r3;\n\t"                                                    \
    "setp.eq.and.u32 pq, r2, r10, pv;\n\t"              /* slot 0 is written to the mirror as well */          \
    "@pq cp.async.cg.shared.global [r5+1536], [rb], 16, r3;\n\t"                                               \
    "cp.async.commit_group;\n\t"                                                                               \
    "add.cc.u32 r11, r11, 512;\n\t"                                                                            \
    "addc.u32 r12, r12, 0;\n\t"                                                                                \
    "sub.s32 r1, r1, 512;\n\t"                                                                                 \
    "add.u32 r2, r2, 512;\n\t"                                                                                 \
    "sub.u32 r4, r2, r10;\n\t"                                                                                 \
    "setp.ge.u32 pv, r4, 1536;\n\t"                                                                            \
    "selp.b32 r2, r10, r2, pv;\n\t"                                                                            \
    "st.shared.v4.u32 [" EP_CTX "+32], {r11, r12, r1, r2};\n\t"                                                       \
    "cp.async.wait_group 1;\n\t"                                                                               \
    "bar.warp.sync 0xffffffff;\n\t"                                                                            \
    "add.u32 wthrA, wthrA, 512;\n\t"            /* the cursor's chunk is the next slot's */                           \
    "sub.u32 r4, wthrA, r10;\n\t"                                                                                     \
    "setp.lt.u32 pq, r4, 2046;\n\t"                                                                            \
    "@pq bra.uni EP_SVC_END_A;\n\t"                                                                                   \
    "sub.u32 wthrA, wthrA, 1536;\n\t"           /* past the third slot: everything back by the ring */                \
    "sub.u32 %1, %1, 1536;\n\t"                                                                                       \
    "ld.shared.u32 r5, [" EP_CTX "+32+20];\n\t"                                                                       \
    "sub.u32 r5, r5, 1536;\n\t"                                                                                \
    "st.shared.u32 [" EP_CTX "+32+20], r5;\n\t"                                                                       \
    "EP_SVC_END_A:\n\t"

#define EP_TILES_LOOP_ASM(BODY, CVT, STORE, GROUP_BYTES)                                                                    \
    asm volatile(                                                                                                     \
        "{\n\t"                                                                                                       \
        EP_REGS                                                                                                       \
        ".reg .pred pq, pv, pr;\n\t"                                                                                  \
        ".reg .b32 r0, r1, r2, r3, r4, r5, r6, r7, r8, r9, r10, r11, r12, c0r, c1r, d0r, d1r, hotb, hotb1;\n\t" \
        ".reg .b64 ra, rb, l2b1;\n\t"                                                                                 \
        ".reg .f32 k0f, k1f;\n\t"                                                                                     \
        "mov.b64 {k0f, k1f}, " EP_KK ";\n\t"                                                                          \
        "mov.b32 c0r, 0x45800000;\n\t"                                                                                \
        "mov.b32 c1r, 0x45800400;\n\t"                                                                                \
        "mov.b32 d0r, 0x4A800000;\n\t"                /* 2^22, 2^22 + 1/2 (2^12-slot streams) */                    \
        "mov.b32 d1r, 0x4A800001;\n\t"                                                                                \
        "add.u32 hotb, " EP_LUT0 ", " EP_HOTOFF ";\n\t"   /* 2^12-slot streams: hot entries of coset 0, */              \
        "add.u32 hotb1, hotb, 16896;\n\t"                 /* of coset 1; complete array of coset 1 */                   \
        "add.s64 l2b1, " EP_L2B ", 131072;\n\t"                                                                       \
        EP_INIT                                                                                                       \
        "bra.uni EP_RARE;\n\t"                                                                                        \
        "EP_LOOP:\n\t"                                                                                                \
        BODY(CVT)                                                                                                     \
        EP_ADDR STORE                                                                                                 \
        EP_ADVANCE(#GROUP_BYTES)                                                                                      \
        /* one vote for everything rare */                                                                            \
        EP_CALM_ALL                                                                                                   \
        "vote.sync.all.pred pq, pq, 0xffffffff;\n\t"                                                                  \
        "@pq bra.uni EP_LOOP;\n\t"                                                                                    \
        "EP_RARE:\n\t"                                                                                                \
        EP_ROWS                                                                                                       \
        "setp.lt.u32 pr, " EP_LT ", 0;\n\t"          /* false */                                                                                   \
        EP_ANY_ACT                                                                                                    \
        "vote.sync.any.pred pr, pr, 0xffffffff;\n\t"                                                                  \
        "@!pr bra.uni EP_DONE;\n\t"                                                                                   \
        EP_SERVICE                                                                                                    \
        "bra.uni EP_LOOP;\n\t"                                                                                        \
        "EP_DONE:\n\t"                                                                                                \
        "}"                                                                                                           \
        /* every read-write operand is early-clobber: the loop reads the inputs after it has updated them */         \
        : "+&r"(x), "+&r"(a), "+&r"(bal), "+&r"(doff)                                                                 \
        : "r"(lt), "r"(lut_addr), "r"(lut_addr + kCosetStride), "r"(ctx), "l"(kk), "l"(out_base), "r"(cf.f0),         \
          "r"(cf.f1), "r"(lane16), "l"(l2base), "r"(hs2), "n"(kHotBase)                                             \
        : "memory")

// ---- the loop for few tiles per SM: one tile per warp, its whole payload in shared memory ---------------------------
// Nothing else covers a warp's stalls here, so the rare work is kept short as well: no ring to refill, and the tile's row
// scales are in shared memory too (a load from global memory at a row's start: 700 cycles every C / 256 groups).
// FULL and REDO are for EP_BODY11_GUESS: a tile's last group, if not every lane has a block in it, and a group whose guess
// failed (stored over) are decoded by EP_BODY11_SHORT.
#define EP_GUESS_TEST "setp.ge.and.u32 pq, lm, 32768, pq;\n\t"
// all lanes have a block, or the other body
#define EP_GUESS_FULL "vote.sync.all.pred pr, actA, 0xffffffff;\n\t" "@!pr bra.uni EP_OTHER;\n\t"
#define EP_GUESS_REDO(CVT, STORE, GROUP_BYTES)                                                                        \
        "setp.lt.u32 pr, lm, 32768;\n\t"                                                                              \
        "vote.sync.any.pred pr, pr, 0xffffffff;\n\t"                                                                  \
        "@!pr bra.uni EP_RARE;\n\t"                                                                                   \
        "mov.b32 %0, sx;\n\t" "mov.b32 %1, sa;\n\t" "mov.b32 %2, sb;\n\t" "sub.u32 %3, %3, " #GROUP_BYTES ";\n\t"     \
        "EP_OTHER:\n\t"                                                                                               \
        EP_BODY11_SHORT(CVT) EP_SHORT_FIN                                                                             \
        EP_ADDR STORE EP_ADVANCE(#GROUP_BYTES)
#define EP_REDO_NONE(CVT, STORE, GROUP_BYTES)
#define EP_FEW_LOOP_ASM(BODY, FIN, INIT, FULL, TEST, REDO, KEEP, CVT, STORE, GROUP_BYTES)                             \
    asm volatile(                                                                                                     \
        "{\n\t"                                                                                                       \
        EP_REGS                                                                                                       \
        ".reg .pred pq, pv, pr, ps;\n\t"                                                                              \
        ".reg .b32 r0, r1, r2, r3, r4, r5, r6, r7, r10, r11, r12, c0r, c1r, lm, sx, sa, sb, ea, va, f2, b2, q2, rp, rowb, endo;\n\t"     \
        ".reg .b64 ra, rb;\n\t"                                                                                       \
        ".reg .f32 k0f, k1f;\n\t"                                                                                     \
        "mov.b64 {k0f, k1f}, " EP_KK ";\n\t"                                                                          \
        "mov.b32 c0r, 0x45800000;\n\t"                                                                                \
        "mov.b32 c1r, 0x45800400;\n\t"                                                                                \
        INIT                                                                                                          \
        "mov.b32 rp, %12;\n\t" "mov.b32 limA, %13;\n\t" "mov.b32 wthrA, %14;\n\t"                                     \
        "ld.shared.b32 sgA, [rp];\n\t" "mov.b32 r3, sgA;\n\t" "mov.b64 ssA, {r3, r3};\n\t"                            \
        "ld.shared.u32 rowb, [" EP_CTX "+8];\n\t"                                                                     \
        "ld.shared.u32 endo, [" EP_CTX "+56];\n\t"        /* offset after the tile's last block */                    \
        "setp.lt.u32 actA, %3, endo;\n\t" "@!actA mov.u32 limA, 0xffffffff;\n\t"                                      \
        "vote.sync.any.pred pr, actA, 0xffffffff;\n\t"                                                                \
        "@!pr bra.uni EP_DONE;\n\t"                                                                                   \
        FULL                                                                                                          \
        "EP_LOOP:\n\t"                                                                                                \
        BODY(CVT)                                                                                                     \
        EP_ADDR STORE EP_ADVANCE(#GROUP_BYTES)                                                                        \
        EP_CALM_ALL                                                                                                   \
        TEST                                                                                                          \
        "vote.sync.all.pred pq, pq, 0xffffffff;\n\t"                                                                  \
        FIN                                                                                                           \
        "@pq bra.uni EP_LOOP;\n\t"                                                                                    \
        REDO(CVT, STORE, GROUP_BYTES)                                                                                 \
        "EP_RARE:\n\t"                                                                                                \
        /* lanes that reached their lim: into the next row (rows hold 32 blocks or more), or past the tile's last block */ \
        "setp.ge.u32 pv, %3, limA;\n\t"                                                                               \
        "vote.sync.any.pred pr, pv, 0xffffffff;\n\t"                                                                  \
        "@!pr bra.uni EP_ROWS_END;\n\t"                                                                               \
        "setp.lt.u32 actA, %3, endo;\n\t"                                                                             \
        "@pv add.u32 rp, rp, 4;\n\t" "ld.shared.b32 sgA, [rp];\n\t" "@pv add.u32 limA, limA, rowb;\n\t"               \
        "min.u32 limA, limA, endo;\n\t" "@!actA mov.u32 limA, 0xffffffff;\n\t"                                        \
        "mov.b32 r3, sgA;\n\t" "mov.b64 ssA, {r3, r3};\n\t"                                                           \
        "vote.sync.any.pred pr, actA, 0xffffffff;\n\t"                                                                \
        "@!pr bra.uni EP_DONE;\n\t"                                                                                   \
        "EP_ROWS_END:\n\t"                                                                                            \
        "setp.ge.u32 pr, %1, wthrA;\n\t"                                                                              \
        "vote.sync.any.pred pr, pr, 0xffffffff;\n\t"                                                                  \
        "@!pr bra.uni EP_WINDOW_END;\n\t"                                                                             \
        /* the cursor reached what was still on its way when the loop began */                                        \
        "cp.async.wait_group 0;\n\t"                                                                                  \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "ld.shared.v4.u32 {r11, r12, r1, r2}, [" EP_CTX "+32];\n\t"   /* source of the window, bytes from there, limit */ \
        "ld.shared.v2.u32 {r10, r5}, [" EP_CTX "+48];\n\t"            /* window, address of position 0 */             \
        "setp.lt.u32 pq, wthrA, r2;\n\t"                                                                              \
        "mov.b32 wthrA, r2;\n\t"                                                                                      \
        "@pq bra.uni EP_WINDOW_END;\n\t"                                                                              \
        /* or the window's end: the window moves on to the cursor (lane 0's address is the lowest), and all of it is copied */ \
        "shfl.sync.idx.b32 r3, %1, 0, 31, 0xffffffff;\n\t"                                                            \
        "sub.u32 r3, r3, r10;\n\t" "and.b32 r3, r3, 0xfffffff0;\n\t"                                                  \
        "sub.u32 %1, %1, r3;\n\t" "sub.u32 r5, r5, r3;\n\t" "sub.s32 r1, r1, r3;\n\t"                                 \
        "add.cc.u32 r11, r11, r3;\n\t" "addc.u32 r12, r12, 0;\n\t" "mov.b64 ra, {r11, r12};\n\t"                      \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "st.shared.v2.u32 [" EP_CTX "+32], {r11, r12};\n\t" "st.shared.u32 [" EP_CTX "+40], r1;\n\t"                  \
        "st.shared.u32 [" EP_CTX "+52], r5;\n\t"                                                                      \
        "mov.b32 r0, " EP_LT ";\n\t" "popc.b32 r0, r0;\n\t" "shl.b32 r0, r0, 4;\n\t"      /* 16 * lane */             \
        "sub.u32 r4, r2, r10;\n\t" "add.u32 r4, r4, 512;\n\t"                             /* the window's size */     \
        "EP_FILL:\n\t"                                                                                                \
        "sub.s32 r6, r1, r0;\n\t" "min.s32 r6, r6, 16;\n\t" "setp.gt.s32 pv, r6, 0;\n\t"                              \
        "setp.lt.and.u32 pv, r0, r4, pv;\n\t"                                                                         \
        "mad.wide.u32 rb, r0, 1, ra;\n\t" "add.u32 r7, r10, r0;\n\t"                                                  \
        "@pv cp.async.cg.shared.global [r7], [rb], 16, r6;\n\t"                                                       \
        "add.u32 r0, r0, 512;\n\t"                                                                                    \
        "vote.sync.any.pred pv, pv, 0xffffffff;\n\t"                                                                  \
        "@pv bra.uni EP_FILL;\n\t"                                                                                    \
        "cp.async.wait_all;\n\t"                                                                                      \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "EP_WINDOW_END:\n\t"                                                                                          \
        FULL                                                                                                          \
        "bra.uni EP_LOOP;\n\t"                                                                                        \
        "EP_DONE:\n\t" KEEP                                                                                           \
        "}"                                                                                                           \
        : "+&r"(x), "+&r"(a), "+&r"(bal), "+&r"(doff)                                                                 \
        : "r"(lt), "r"(lut_addr), "r"(lut_addr + kCosetStride), "r"(ctx), "l"(kk), "l"(out_base), "r"(cf.f0), "r"(cf.f1), \
          "r"(rp), "r"(lim), "r"(wthr)                                                                                \
        : "memory")

#define EP_FEW_GUESS_ASM(BODY, REGS, KEEP, CVT, STORE, GROUP_BYTES)                                                   \
    EP_FEW_LOOP_ASM(BODY, EP_GUESS_FIN, REGS EP_GUESS_INIT, EP_GUESS_FULL, EP_GUESS_TEST, EP_GUESS_REDO, KEEP, CVT, STORE, GROUP_BYTES)

// One tile of a tensor whose rows hold at least 32 blocks and whose tables have 2^B slots (B = 11: one-level tables; B = 12: two
// levels, see EP_N1).  A warp whose slot lies past the job's last tile gets that last tile's record, only so that its addresses
// stay inside the stream, and no block at all.  The number of groups is data here, not control flow the compiler
// reasons about: every branch on it is a bra.uni on a warp vote.
// `tables`: the job's lookup tables may still be being written (by this CTA's own stores or copies): the
// tile's record and first payload chunks are requested first, the wait comes after.
template <int DT, int B>
__device__ __forceinline__ void decode_tile_fast(const JobParams &J, uint32_t first, uint32_t tiles_per_round, uint32_t lut_addr,
                                                  CosetFreq cf, uint32_t ring, uint32_t ctx, uint32_t lane, const TablesWait &tables) {
    constexpr uint32_t BB = Out<DT>::kBlockBytes;
    const uint32_t lt = (1u << lane) - 1u, lane16 = 16u * lane;
    // (a warp without a tile in this round - the job's last round, or a CTA with more warps than tiles - has no block)
    const bool valid = first < J.tile_cnt && (threadIdx.x >> 5) < tiles_per_round;
    const uint32_t tile = J.tile0 + min(first, J.tile_cnt - 1u), cctx = ctx + kCtxChain;
    const TileSetup T = tile_setup(J, tile, valid, lane);
    for (uint32_t k = 0; k < kRingSlots; ++k) ring_issue(ring, T.a0, T.room, k, lane);
    // the record of the tile this warp takes in the CTA's next round (132 bytes: two lines), into L2
    if (lane < 2u && tile + tiles_per_round < J.n_tiles) prefetch_l2(J.tile_index + size_t(tile + tiles_per_round) * 33u + 32u * lane);
    if (lane == 0) {                 // the next request is chunk 3, into slot 0
        prefetch_l2(J.scales + min(T.v0 / J.per_row, J.row_max));      // the first row scale the loop will ask for
        sts64(cctx + kCcSrc, T.a0 + kRingBytes);
        sts32(cctx + kCcRem, T.room - kRingBytes);
        sts32(cctx + kCcDst, ring);
        sts32(cctx + kCcRing, ring);
        sts32(cctx + kCcWbase, ring);
        sts32(cctx + kCcEndo, (T.v0 + T.nv) * BB);
    }
    uint32_t x = T.x, a = ring + T.lead, bal = 0, doff = (T.v0 + lane) * BB;
    cp_async_wait<1>();           // all but the third chunk have landed
    __syncwarp();
    wait_for_tables(tables);
    const uint32_t k0 = __float_as_uint(float((B == 11 ? 4096 : 4194304) - J.zlo));
    const uint64_t kk = pack64(k0, k0);
    const uint64_t out_base = reinterpret_cast<uint64_t>(J.out);
    const uint64_t l2base = reinterpret_cast<uint64_t>(J.cold);
    const uint32_t hs2 = J.hs2;
    if constexpr (B == 11) {
        if constexpr (DT == EP_BF16) EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_BF16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP16) EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_FP16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP8_E4M3) EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_E4M3, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP8_E5M2) EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_E5M2, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP32) EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_FP32, EP_ST_FP32, 1024);
        else if constexpr (DT == EP_UINT8) EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_I8, EP_ST_UINT8, 256);
        else EP_TILES_LOOP_ASM(EP_BODY11, EP_CVT_I8, EP_ST_INT8, 256);
    } else {
        if constexpr (DT == EP_BF16) EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_BF16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP16) EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_FP16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP8_E4M3) EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_E4M3, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP8_E5M2) EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_E5M2, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP32) EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_FP32, EP_ST_FP32, 1024);
        else if constexpr (DT == EP_UINT8) EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_I8, EP_ST_UINT8, 256);
        else EP_TILES_LOOP_ASM(EP_BODY12, EP_CVT_I8, EP_ST_INT8, 256);
    }
    cp_async_wait<0>();           // nothing may still be landing in the ring when the next tile starts
    __syncwarp();
    // integrity: the encoder started every state at 2^15 and a tile's words end where the next tile's begin
    const uint32_t cur = __shfl_sync(0xFFFFFFFFu, a, 0) + 2u * __popc(bal) - lds32(cctx + kCcWbase);
    const bool bad = valid && ((x != ep::kStateLow) || (T.off + ((cur - T.lead) >> 1) != T.end));
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&g_ep_status, 1u);
    __syncwarp();                 // the context block is rewritten by the next tile
}

// One tile of a CTA that has few of them (2^11-slot streams, rows of 32 blocks or more), decoded by the loop that is short in
// latency, not in instructions.  The tiles of a round share the space of the 32 rings and of the hot window: 6 KB for each
// of sixteen, 12 KB for each of eight, which holds a tile's row scales and, usually, all of its payload.  (As in decode_tile_fast every branch
// depends on parameters or is a bra.uni on a vote: a guard around each vote would cost 25 cycles.)
template <int DT>
__device__ __forceinline__ void decode_tile_few(const JobParams &J, uint32_t first, uint32_t tiles_per_round, uint32_t lut_addr,
                                                CosetFreq cf, uint32_t ctx, uint32_t lane, const TablesWait &tables) {
    constexpr uint32_t BB = Out<DT>::kBlockBytes, kHead = 1024;
    const uint32_t warp = threadIdx.x >> 5, space = kStageBytes / tiles_per_round & ~127u;
    const bool valid = first < J.tile_cnt && warp < tiles_per_round;
    const uint32_t scales = lut_addr + kRingBase + min(warp, tiles_per_round - 1u) * space;   // row scales, then the window
    const uint32_t tile = J.tile0 + min(first, J.tile_cnt - 1u);
    const TileSetup T = tile_setup(J, tile, valid, lane);
    const uint32_t row0 = T.v0 / J.per_row, rows = valid ? (T.v0 + T.nv - 1u) / J.per_row - row0 + 1u : 0u;
    const uint32_t scale_bytes = (4u * ((J.V + J.per_row - 1u) / J.per_row + 2u) + 127u) & ~127u;    // (checked by the launcher)
    const uint32_t window = scales + scale_bytes, size = space - scale_bytes;
    const uint32_t bytes = valid ? min(T.lead + 2u * (min(T.end, J.total_words) - min(T.off, T.end)), size) : 0u;
    // the scales and the first kilobyte, then the rest, as two groups of copies
    for (uint32_t i = lane; i < rows; i += 32u)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(scales + 4u * i), "l"(J.scales + row0 + i) : "memory");
    for (uint32_t o = 16u * lane; o < min(bytes, kHead); o += 512u)
        cp_async16(window + o, T.a0 + (o < T.room ? o : 0u), o < T.room ? min(16u, T.room - o) : 0u);
    cp_async_commit();
    for (uint32_t o = kHead + 16u * lane; o < bytes; o += 512u)
        cp_async16(window + o, T.a0 + (o < T.room ? o : 0u), o < T.room ? min(16u, T.room - o) : 0u);
    cp_async_commit();
    uint32_t x = T.x, a = window + T.lead, bal = 0, doff = (T.v0 + lane) * BB;
    const uint32_t endo = (T.v0 + T.nv) * BB;
    const uint32_t row = min(T.v0 + lane, T.v0 + max(T.nv, 1u) - 1u) / J.per_row;
    const uint32_t rp = scales + 4u * (row - row0), lim = min((row + 1u) * J.row_bytes, endo);
    // a group reads at most 510 bytes from the cursor on
    const uint32_t limit = window + size - 512u, wthr = bytes > kHead ? window + kHead - 512u : limit;
    if (lane == 0 && warp < tiles_per_round) {
        sts64(ctx + kCtxChain + kCcSrc, T.a0);
        sts32(ctx + kCtxChain + kCcRem, T.room);
        sts32(ctx + kCtxChain + kCcDst, limit);
        sts32(ctx + kCtxChain + kCcRing, window);
        sts32(ctx + kCtxChain + kCcWbase, window);
    }
    if (lane == 0) sts32(ctx + kCtxChain + kCcEndo, endo);
    cp_async_wait<1>();           // the scales and the first kilobyte
    __syncwarp();
    wait_for_tables(tables);
    const uint32_t k0 = __float_as_uint(float(4096 - J.zlo)), lt = (1u << lane) - 1u;
    const uint64_t kk = pack64(k0, k0), out_base = reinterpret_cast<uint64_t>(J.out);
    if (J.guess) {
        if constexpr (DT == EP_BF16) EP_FEW_GUESS_ASM(EP_BODY11_GUESS16, "", "", EP_CVT_BF16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP16) EP_FEW_GUESS_ASM(EP_BODY11_GUESS16, "", "", EP_CVT_FP16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP8_E4M3) EP_FEW_GUESS_ASM(EP_BODY11_GUESS8, EP_K8_REGS, EP_K8_KEEP, EP_CVT_E4M3, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP8_E5M2) EP_FEW_GUESS_ASM(EP_BODY11_GUESS8, EP_K8_REGS, EP_K8_KEEP, EP_CVT_E5M2, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP32) EP_FEW_GUESS_ASM(EP_BODY11_GUESS32, "", "", EP_CVT_FP32, EP_ST_FP32, 1024);
        else if constexpr (DT == EP_UINT8) EP_FEW_GUESS_ASM(EP_BODY11_GUESS8, EP_K8_REGS, EP_K8_KEEP, EP_CVT_I8, EP_ST_UINT8, 256);
        else EP_FEW_GUESS_ASM(EP_BODY11_GUESS8, EP_K8_REGS, EP_K8_KEEP, EP_CVT_I8, EP_ST_INT8, 256);
    } else {
        if constexpr (DT == EP_BF16) EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_BF16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP16) EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_FP16, EP_ST_16, 512);
        else if constexpr (DT == EP_FP8_E4M3) EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_E4M3, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP8_E5M2) EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_E5M2, EP_ST_F8, 256);
        else if constexpr (DT == EP_FP32) EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_FP32, EP_ST_FP32, 1024);
        else if constexpr (DT == EP_UINT8) EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_I8, EP_ST_UINT8, 256);
        else EP_FEW_LOOP_ASM(EP_BODY11_SHORT, EP_SHORT_FIN, "", "", "", EP_REDO_NONE, "", EP_CVT_I8, EP_ST_INT8, 256);
    }
    cp_async_wait<0>();           // nothing may still be landing in the stage when the next tile starts
    __syncwarp();
    const uint32_t cur = __shfl_sync(0xFFFFFFFFu, a, 0) + 2u * __popc(bal) - lds32(ctx + kCtxChain + kCcWbase);
    const bool bad = valid && ((x != ep::kStateLow) || (T.off + ((cur - T.lead) >> 1) != T.end));
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&g_ep_status, 1u);
    __syncwarp();
}

// One persistent CTA per SM.  The rounds of all jobs of the launch form one list (job after job); CTA k takes the
// rounds whose cumulative cost at their start lies in [k, k + 1) * ceil(total / gridDim.x) - a contiguous stretch,
// usually inside one job - and sets the lookup tables up again when the stretch crosses into the next job.  Everything
// that steers this (loop bounds, job changes) depends on blockIdx and kernel parameters only, so the compiler
// sees warp-uniform control flow and puts no divergence guards around the warp votes of the hot loop; in the last
// round of a job a warp past the job's last tile goes through the same code with no block to decode.
// FEW: launches of few tiles per CTA (see decode_tile_few); a kernel of its own because it may use 128 registers where 32 warps
// leave 64.
template <int DT, bool FEW>
__global__ void __launch_bounds__(FEW ? 32 * (kFewTiles > kMinWarps ? kFewTiles : kMinWarps) : kThreads, 1)
ep_decode_smem_kernel(const __grid_constant__ BatchParams P) {
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t lut_addr = uint32_t(__cvta_generic_to_shared(smem));
    const uint32_t ring = lut_addr + kRingBase + warp * kRingStride;
    const uint32_t ctx = lut_addr + kCtxBase + warp * kCtxBytes;
    // The hot loop's 64 registers have no room for a phase and a flag kept from job to job, so there every job has an mbarrier of its
    // own (block of seven at 2.5 bpp to FP8 303.5 -> 299.7 us, 8192 x 8192 at 8 bpp 101.1 -> 100.1).  With few tiles per CTA one
    // mbarrier and its phase are the faster way (4096 x 4096 at 3 bpp 38.4 us, 39.1 with one per job).
    bool tables_in_use = false;
    TablesWait tables{kTablesThere, lut_addr + kCtxBase + kCtxTablesBar, FEW ? 1u : 0u};
    if (threadIdx.x == 0) {
        for (int j = 0; j < (FEW ? 1 : P.n_jobs); ++j) mbar_init(lut_addr + kCtxBase + kCtxTablesBar + j * kCtxBytes, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    wait_for_stream();
    for (int j = 0; j < P.n_jobs; ++j) {
        const JobParams &J = P.job[j];
        // rounds r of this job with cost_begin + r * round_cost in [lo, hi), this CTA's share of the total cost
        // (recomputed per job rather than kept in registers across the decode loops)
        const uint32_t lo = P.cost_per_cta * blockIdx.x, hi = lo + P.cost_per_cta;      // below 2^31 (see the launcher)
        const uint32_t a = lo > J.cost_begin ? lo - J.cost_begin : 0u, b = hi > J.cost_begin ? hi - J.cost_begin : 0u;
        const uint32_t r0 = min((a + J.round_cost - 1u) / J.round_cost, J.rounds);
        const uint32_t r1 = min((b + J.round_cost - 1u) / J.round_cost, J.rounds);
        if (r0 >= r1) continue;
        const bool again = FEW ? tables_in_use : lo < J.cost_begin;     // (may also be set for a CTA's first job there)
        if (again) __syncthreads();                  // every warp is done with the previous job's tables
        // the table image is requested first: the tiles' records and payload (two dependent reads of memory that no
        // cache holds yet) are on their way while it arrives
        if (J.lut_image) {
            tables.pending = kTablesCopied;
            if constexpr (FEW) tables.parity ^= 1u;
            else tables.bar = lut_addr + kCtxBase + kCtxTablesBar + j * kCtxBytes;
            if (threadIdx.x == 0) {
                if (again) fence_async_smem();           // the last job's lookups, ordered before this by the barrier above
                copy_tables_smem(J.lut_image, lut_addr, tables.bar, J.b == 12u);
            }
        } else {
            tables.pending = kTablesBuilt;
            build_tables_smem(J, lut_addr, warp, lane);
        }
        const CosetFreq cf = load_coset(J);
        tables_in_use = true;
        // (a stream with 2^12 slots reaches this kernel only in the configuration of the hot loop: see the launcher)
        const bool fast = DT != EP_FIELDS_I32 && J.per_row >= 32u && (J.b == 11u || J.b == 12u) && J.V < (1u << 20);
        if (fast && lane == 0) {                     // what the hot loop's rare paths need to know about the job
            sts64(ctx + kCtxScales, reinterpret_cast<uint64_t>(J.scales));
            sts32(ctx + kCtxRowBytes, J.row_bytes);
            sts32(ctx + kCtxRowMax, J.row_max);      // the step after a tensor's last block must not read past the scales
            sts32(ctx + kCtxRowRcp, J.row_rcp);
        }
        __syncwarp();
        for (uint32_t r = r0; r < r1; ++r) {
            const uint32_t base = r * P.tiles_per_round + warp;
            if constexpr (DT != EP_FIELDS_I32) {
                if (fast) {
                    if (J.b == 12u) {
                        decode_tile_fast<DT, 12>(J, base, P.tiles_per_round, lut_addr, cf, ring, ctx, lane, tables);
                    } else if constexpr (FEW) {
                        decode_tile_few<DT>(J, base, P.tiles_per_round, lut_addr, cf, ctx, lane, tables);
                    } else {
                        decode_tile_fast<DT, 11>(J, base, P.tiles_per_round, lut_addr, cf, ring, ctx, lane, tables);
                    }
                    tables.pending = kTablesThere;
                    continue;
                }
            }
            wait_for_tables(tables);
            tables.pending = kTablesThere;
            if (base < J.tile_cnt && warp < P.tiles_per_round) decode_tile_plain<DT>(J, J.tile0 + base, lut_addr, cf, ring, lane);
        }
    }
}

// ======================================================================================================
// Decode fused into a matrix product (the step the paper leaves as future work, Sec. "Limitations and future
// work": its decoder still materialises the dense tensor before the product).  First slice: y = x W^T for up
// to 32 tokens - the regime in which reading the weights dominates a linear layer -, W decoded tile by tile
// straight into the shared-memory operand of a tcgen05 matrix instruction and never written to global memory.
//
// The stream must have one tile per row of W (V = C / 8) and C a multiple of 256.  The rows are spread evenly over
// the SMs; a CTA takes its range in equal steps of at most 30 rows, one row per warp: warps 2 .. decode their rows group by
// group (a group = 32 blocks = 256 columns), so after every group the CTA holds a 30 x 256 slab of W - the B operand
// (N = 32, K-major, 128-byte swizzle: a lane's 16-byte block is one piece of a swizzled row, so
// the stores are conflict-free).  Warps 0 and 1 decode nothing.  One lane of warp 0 brings the matching 256
// columns of x in (A operand, M = 64 rows of which the first 16 or 32 are tokens; the others read whatever shared
// memory follows and produce accumulator rows nobody stores) with four tensor copies (cp.async.bulk.tensor, the
// copy engine swizzles).  One lane of warp 1 waits until x has landed and all rows of the slab are stored and
// issues the slab's sixteen K = 16 instructions.  (A decoding warp cannot do that on the side: whoever issues falls
// behind by the time it takes, and with two slabs every warp is at most one group ahead of the slowest - measured
// 138 us for the 10240 x 3840 layer; one warp for copies and instructions together 90 us, its single instruction stream
// being the slowest in the CTA.)  The fp32 accumulator (64 lanes x 32 columns) stays in tensor memory over the whole row;
// there are two, used in turn, and warps 0 and 1 - whose quarters of tensor memory hold the tokens - read one out while the
// decoding warps are in the next step: nothing holds those up between steps.
// 10240 x 3840, 16 tokens: steps of 30 + 30 + 10 rows, each ended by a CTA barrier around the read-out, the group in C++:
// 74.3 us.
//
// Shared memory: the lookup tables (128 KB), a payload ring of 4 x 256 + 512 or 3 x 512 + 512 bytes for each decoding warp, then A (units
// of x, refilled by the loading warp as soon as the instructions that read them are done), B (two slabs: the warps decode
// the next group while the tensor core reads the last one) and the mbarriers; see GemmShape.  What bounds the token count:
// a group's columns of x must be in flight while the group is decoded (about 1 us), and every CTA re-reads x from L2.
// Every wait on an mbarrier gives up after kSpinLimit polls, raises the abort word and lets the kernel run to its
// end (wrong output, status flag set) instead of hanging.
struct GemmParams {
    JobParams J;
    float *y;                     // [T, R] fp32, row-major
    uint32_t T, Tpad;             // tokens; rows of x that are staged (16 or 32)
    uint32_t R;
    uint32_t rows_per_cta;        // CTA k takes rows [k, k + 1) * rows_per_cta,
    uint32_t rows_per_step, steps;   // rows_per_step at a time
    uint32_t groups;              // C / 256
};

// What depends on the rows per step.  Thirty leave 16 KB for x: two units of a whole group for up to 16 tokens, of half a group
// for up to 32, and then a unit can be asked for only when the instructions half a group before have read it, and payload rings
// of 4 x 256 bytes.  24 rows make room for 16 KB more: for up to 32 tokens four units of half a group each, for up to 16 (whose
// two units are enough) rings of 3 x 512 bytes, which are served half as often: 27 of 250 instructions per group were the ring's.
// 4 bpp, 16 tokens, us, 4 x 256 / 3 x 512: 70 rows per SM of 3840 columns 53.4 / 51.9, 31 of 2048 19.6 / 19.0, 23 at 5 bpp
// 13.4 / 13.1.  Where 24 rows take more steps than thirty they are the slower ones (see the launcher).
template <uint32_t TPAD, uint32_t ROWS>
struct GemmShape {
    static constexpr bool kWide = TPAD == 16 && ROWS <= 24;
    static constexpr uint32_t kChunk = kWide ? 512 : 256, kSlots = kWide ? 3 : 4, kRing = kChunk * kSlots;   // payload ring of a decoding warp
    static constexpr uint32_t kRingStride = kRing + kRingMirror;
    static constexpr uint32_t kRows = ROWS;                              // most rows of W per step: one per decoding warp
    static constexpr uint32_t kN = (ROWS + 7u) & ~7u;                    // rows of the B operand
    static constexpr uint32_t kUnits = TPAD == 16 || ROWS > 24 ? 2 : 4;                // units of x, 8 KB each
    static constexpr uint32_t kBTile = kN * 128, kSlab = 4 * kBTile;     // B: per slab four 64-column tiles of kN rows
    static constexpr uint32_t kA = (kRingBase + kRows * kRingStride + 1023u) & ~1023u;   // A operand (swizzled tiles start on 1024-byte boundaries)
    static constexpr uint32_t kB = kA + kUnits * 8192;
    static constexpr uint32_t kBar = kB + 2 * kSlab;                     // mbarriers, tensor-memory address, abort word
    static constexpr uint32_t kSmem = kBar + 256;
    static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kN >> 3) << 17) | ((64u >> 4) << 24);   // f32 += bf16 x bf16, K-major both, N = kN, M = 64
    static_assert(kSmem <= 232448, "more shared memory than an sm_100 CTA can have");
    // a group begins before its chunk's last two bytes and reads 510 bytes at most: all chunks but the newest hold them, behind the
    // ring's end the mirror does
    static_assert((kSlots - 1u) * kChunk >= kChunk - 2u + 510u && kRingMirror >= 510u && kRingMirror % kChunk == 0);
};

// a test that never waits
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// one attempt: the thread may be suspended by the hardware for up to about a microsecond while the phase is pending
// (a busy test_wait loop of 32 waiting lanes took half of the kernel's issue slots away from the decoding warps)
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(1000u) : "memory");
    return ok != 0;
}
// waits for the phase of the given parity to complete; false (and the abort word set) if it does not within the limit
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t abort_addr) {
    if (mbar_test(bar, parity)) return true;             // usually the phase is long complete
    if (lds32(abort_addr)) return false;
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 255u) == 255u && lds32(abort_addr)) return false;
    }
    sts32(abort_addr, 1u);
    return false;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// K-major operand tile with 128-byte swizzle: rows of 128 bytes, groups of eight rows 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
    return uint64_t((smem_addr >> 4) & 0x3FFFu) | (uint64_t(1) << 16) | (uint64_t(1024 >> 4) << 32) | (uint64_t(1) << 46) |
           (uint64_t(2) << 61);
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// A row's groups (BODY) with operands of its own: %0 .. %3 = x, a, bal and the group counter q, which goes on from
// row to row.  In C++ around a group's asm this took 324 instructions per group, 80 of them guards around the votes and 40
// for the ring; thirty warps are bound by just that number.
// Per group: is the slab free, i.e. is the tensor core done with the group two before (tested ahead of the decode; a fresh
// barrier passes for parity 1)?  Decode, wait if need be (kSpinLimit tries, or until the abort word is set), store the
// block, arrive; then the ring (EP_SERVICE's steps, for either ring; a group may leave two chunks of 256 bytes).
#undef EP_LT
#undef EP_LUT0
#undef EP_LUT1
#undef EP_CTX
#undef EP_KK
#undef EP_F0
#undef EP_F1
#define EP_LT "%4"
#define EP_LUT0 "%5"
#define EP_LUT1 "%6"
#define EP_CTX "%7"
#define EP_KK "%8"
#define EP_F0 "%9"
#define EP_F1 "%10"
#define EP_GEMM_ROW_ASM(BODY)                                                                                                 \
    asm volatile("{\n\t" EP_REGS                                                                                      \
        ".reg .pred pq, pv, pr, pl;\n\t"                                                                              \
        ".reg .b32 r0, r1, r2, r3, r4, r5, r6, r10, r11, r12, c0r, c1r, g, bar, par, odd, dst, tries;\n\t"   \
        ".reg .b64 ra, rb, st;\n\t"                                                                                   \
        "mov.b32 c0r, 0x45800000;\n\t" "mov.b32 c1r, 0x45800400;\n\t"                \
        "mov.b64 ssA, {%11, %11};\n\t" "setp.ne.u32 actA, %12, 0;\n\t" "mov.b32 g, %13;\n\t"                          \
        "setp.eq.u32 pl, " EP_LT ", 0;\n\t"                  /* lane 0 */                                             \
        "ld.shared.u32 r10, [" EP_CTX "+48];\n\t" "add.u32 wthrA, r10, %19 - 2;\n\t"                                      \
        "EP_LOOP:\n\t"                                                                                                \
        "and.b32 odd, %3, 1;\n\t" "mad.lo.u32 bar, odd, 8, %15;\n\t" "mad.lo.u32 dst, odd, %17, %14;\n\t"             \
        "shr.u32 par, %3, 1;\n\t" "and.b32 par, par, 1;\n\t" "xor.b32 par, par, 1;\n\t"                               \
        "mbarrier.test_wait.parity.shared::cta.b64 pv, [bar], par;\n\t"                                               \
        BODY(EP_CVT_BF16)                                                                                             \
        "vote.sync.all.pred pv, pv, 0xffffffff;\n\t"                                                                  \
        "@pv bra.uni EP_FREE;\n\t"                                                                                    \
        "mov.b32 tries, %18;\n\t"                                                                                     \
        "EP_WAIT:\n\t"                                                                                                \
        "mbarrier.try_wait.parity.shared::cta.b64 pv, [bar], par, 1000;\n\t"                                          \
        "vote.sync.any.pred pv, pv, 0xffffffff;\n\t"                                                                  \
        "@pv bra.uni EP_FREE;\n\t"                                                                                    \
        "ld.volatile.shared.u32 r0, [%16+100];\n\t" "setp.ne.u32 pv, r0, 0;\n\t"          /* the abort word */        \
        "vote.sync.any.pred pv, pv, 0xffffffff;\n\t"                                                                  \
        "@pv bra.uni EP_FREE;\n\t"                                                                                    \
        "sub.u32 tries, tries, 1;\n\t" "setp.ne.u32 pv, tries, 0;\n\t"                                                \
        "vote.sync.any.pred pv, pv, 0xffffffff;\n\t"                                                                  \
        "@pv bra.uni EP_WAIT;\n\t"                                                                                    \
        "mov.b32 r0, 1;\n\t" "st.volatile.shared.u32 [%16+100], r0;\n\t"                                              \
        "EP_FREE:\n\t"                                                                                                \
        "st.shared.v4.b32 [dst], {o0A, o1A, o2A, o3A};\n\t"                                                           \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "mad.lo.u32 bar, odd, 8, %16;\n\t"                                                                            \
        "@pl mbarrier.arrive.shared::cta.b64 st, [bar];\n\t"                                                          \
        "add.u32 %3, %3, 1;\n\t" "sub.u32 g, g, 1;\n\t"                                                               \
        "setp.lt.u32 pq, %1, wthrA;\n\t" "setp.ne.and.u32 pq, g, 0, pq;\n\t"                                          \
        "vote.sync.all.pred pq, pq, 0xffffffff;\n\t"                                                                  \
        "@pq bra.uni EP_LOOP;\n\t"                                                                                    \
        "setp.eq.u32 pr, g, 0;\n\t"                                                                                   \
        "vote.sync.any.pred pr, pr, 0xffffffff;\n\t"                                                                  \
        "@pr bra.uni EP_DONE;\n\t"                                                                                    \
        "EP_RING:\n\t"                                                                                                \
        "shfl.sync.idx.b32 r6, %1, 0, 31, 0xffffffff;\n\t" "popc.b32 r0, %2;\n\t" "mad.lo.u32 r6, r0, 2, r6;\n\t"     \
        "add.u32 r0, wthrA, 2;\n\t" "setp.lt.u32 pq, r6, r0;\n\t"                                                     \
        "vote.sync.all.pred pq, pq, 0xffffffff;\n\t"                                                                  \
        "@pq bra.uni EP_LOOP;\n\t"                           /* the cursor has not left its chunk */                  \
        "ld.shared.v4.u32 {r11, r12, r1, r2}, [" EP_CTX "+32];\n\t"   /* source, bytes left, destination */           \
        "mov.b64 ra, {r11, r12};\n\t"                                                                                 \
        "popc.b32 r4, " EP_LT ";\n\t" "shl.b32 r4, r4, 4;\n\t"        /* 16 * lane */                                 \
        "sub.s32 r3, r1, r4;\n\t" "min.s32 r3, r3, 16;\n\t"                                                           \
        "setp.gt.s32 pv, r3, 0;\n\t" "setp.lt.and.u32 pv, r4, %19, pv;\n\t"                                           \
        "mad.wide.u32 rb, r4, 1, ra;\n\t" "add.u32 r5, r2, r4;\n\t"                                                   \
        "@pv cp.async.cg.shared.global [r5], [rb], 16, r3;\n\t"                                                       \
        "sub.u32 r4, r2, r10;\n\t" "setp.lt.and.u32 pq, r4, 512, pv;\n\t"   /* the ring's first 512 bytes are written to the mirror as well */ \
        "@pq cp.async.cg.shared.global [r5+%20], [rb], 16, r3;\n\t"                                                  \
        "cp.async.commit_group;\n\t"                                                                                  \
        "add.cc.u32 r11, r11, %19;\n\t" "addc.u32 r12, r12, 0;\n\t" "sub.s32 r1, r1, %19;\n\t"                        \
        "add.u32 r2, r2, %19;\n\t" "setp.ge.u32 pv, r4, %20 - %19;\n\t" "selp.b32 r2, r10, r2, pv;\n\t"                     \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "st.shared.v4.u32 [" EP_CTX "+32], {r11, r12, r1, r2};\n\t"                                                   \
        "cp.async.wait_group 1;\n\t"                                                                                  \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "add.u32 wthrA, wthrA, %19;\n\t" "sub.u32 r4, wthrA, r10;\n\t" "setp.lt.u32 pq, r4, %20 + %19 - 2;\n\t"                \
        "vote.sync.all.pred pq, pq, 0xffffffff;\n\t"                                                                  \
        "@pq bra.uni EP_RING;\n\t"                                                                                    \
        "sub.u32 wthrA, wthrA, %20;\n\t" "sub.u32 %1, %1, %20;\n\t"   /* past the last slot: everything back by the ring */ \
        "ld.shared.u32 r5, [" EP_CTX "+52];\n\t" "sub.u32 r5, r5, %20;\n\t"                                           \
        "bar.warp.sync 0xffffffff;\n\t"                                                                               \
        "st.shared.u32 [" EP_CTX "+52], r5;\n\t"                                                                      \
        "bra.uni EP_RING;\n\t"                                                                                        \
        "EP_DONE:\n\t"                                                                                                \
        "}"                                                                                                           \
        : "+&r"(x), "+&r"(a), "+&r"(bal), "+&r"(q)                                                                    \
        : "r"(lt), "r"(lut_addr), "r"(lut_addr + kCosetStride), "r"(ctx), "l"(kk), "r"(cf.f0), "r"(cf.f1), "r"(sigma), "r"(act), \
          "r"(P.groups), "r"(b_dst), "r"(bar_mma), "r"(bar_b), "n"(G::kSlab), "n"(kSpinLimit), "n"(G::kChunk), "n"(G::kRing)                         \
        : "memory")

template <uint32_t TPAD, uint32_t ROWS>
__global__ void __launch_bounds__(kThreads, 1) ep_decode_gemm_kernel(const __grid_constant__ GemmParams P,
                                                                     const __grid_constant__ CUtensorMap x_map) {
    extern __shared__ __align__(16) uint8_t smem[];      // (the operand tiles need 1024: checked at run time, see abort word)
    const JobParams &J = P.J;
    // (the warp's number by a shuffle: the compiler then knows that roles are warp-uniform and puts no guard around each vote
    // of the decoding loop, which cost 500 of 1700 cycles per group)
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const uint32_t lut_addr = uint32_t(__cvta_generic_to_shared(smem));
    using G = GemmShape<TPAD, ROWS>;
    const uint32_t a_base = lut_addr + G::kA, b_base = lut_addr + G::kB;
    // A holds two or four units of x: four tiles of 64 columns x 16 rows each (one group's columns), or two tiles x 32 rows
    // (half a group's).  Per unit one mbarrier "landed" and one "read"; per slab of B one "rows stored" and one "read".
    constexpr uint32_t a_tile_bytes = TPAD * 128u, kUnitTiles = 8192u / a_tile_bytes, kUnitsPerGroup = 4u / kUnitTiles;
    const uint32_t bar_a = lut_addr + G::kBar, bar_afree = bar_a + 64u, bar_mma = bar_a + 128u, bar_b = bar_a + 144u,
                   slot = bar_a + 160u, abort_addr = bar_b + 100u;
    const TablesWait tables{kTablesCopied, bar_a + 168u, 0u};
    if (tid == 0) {
        for (uint32_t i = 0; i < G::kUnits; ++i) {
            mbar_init(bar_a + 8u * i, 1u);       // the loading lane's arrival; completes when the unit's tiles have landed
            mbar_init(bar_afree + 8u * i, 1u);   // the commit after the matrix instructions that read the unit
        }
        for (uint32_t i = 0; i < 2u; ++i) {
            mbar_init(bar_mma + 8u * i, 1u);     // the commit after a group's matrix instructions
            mbar_init(bar_b + 8u * i, P.rows_per_step);   // every decoding warp, when its row of the slab is stored
        }
        mbar_init(tables.bar, 1u);
        sts32(abort_addr, (lut_addr & 1023u) ? 1u : 0u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {                         // 64 columns of tensor memory: two 64 x 32 fp32 accumulators
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(64u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // (rows of the slabs that belong to no warp, or whose warp has no row in a CTA's last step, hold what they hold: they make
    // columns of the accumulator that nobody stores)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    wait_for_stream();
    if (tid == 0) copy_tables_smem(J.lut_image, lut_addr, tables.bar, false);
    const CosetFreq cf = load_coset(J);
    const uint32_t tmem = lds32(slot);

    const uint32_t row_begin = min(blockIdx.x * P.rows_per_cta, P.R), row_end = min(row_begin + P.rows_per_cta, P.R);
    // the accumulator of step s (tokens 16 quarter ..) to y: with M = 64, token 16 w + l is lane l < 16 of warp w's quarter;
    // columns = rows of W
    auto read_out = [&](uint32_t s, uint32_t quarter) {
        tc_fence_after();
        uint32_t v[32];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                     "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, "
                     "%23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
                       "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
                       "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
                       "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                     : "r"(tmem + ((quarter * 32u) << 16) + 32u * (s & 1u)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        tc_fence_before();
        const uint32_t t = quarter * 16u + lane, r0 = row_begin + s * P.rows_per_step;
        if (lane < 16u && t < P.T && r0 < row_end) {
            float *dst = P.y + size_t(t) * P.R + r0;
            const uint32_t n = min(P.rows_per_step, row_end - r0);
#pragma unroll
            for (uint32_t i = 0; i < G::kRows; ++i)
                if (i < n) dst[i] = __uint_as_float(v[i]);
        }
        __syncwarp();
    };
    bool bad = false;
    // unit j of x lies in buffer j mod 2^depth.  (Rows of one group have two half-group units per step: with four buffers the
    // loading warp would be a step too far ahead of the read-out.)
    const uint32_t depth = G::kUnits == 4u && P.groups > 1u ? 2u : 1u, units_mask = (1u << depth) - 1u;

    if (warp == 0) {
        // ---- the loading warp: one lane brings x into A, unit after unit; between two units the warp reads out accumulators ----
        // tile i of the CTA's sequence = columns [64 i, 64 i + 64) of x, counted over all groups (and again from column 0 for
        // every step); the copy engine lays it out and swizzles it; rows past the last token lie outside the tensor and
        // arrive as zeros.  A unit may overwrite the one before it in its buffer when that has been read; where that was a
        // step's last, the step's accumulator is then complete, and it is read out before any unit is loaded that the next
        // user of this accumulator waits for.
        const uint32_t tiles_per_step = 4u * P.groups, units = kUnitsPerGroup * P.groups, total = units * P.steps;
        for (uint32_t j = 0; j < total + units_mask + 1u; ++j) {
            const uint32_t buf = j & units_mask;
            uint32_t go = 1u;
            // (after a wait that ran out nothing is copied any more: re-arming a barrier whose phase never completed
            // would overflow its transaction count)
            if (lane == 0 && j > units_mask) go = mbar_wait(bar_afree + 8u * buf, ((j >> depth) - 1u) & 1u, abort_addr);
            go = __shfl_sync(0xFFFFFFFFu, go, 0);
            if (!go) break;
            if (j > units_mask && (j - units_mask) % units == 0u) read_out((j - units_mask) / units - 1u, 0u);
            if (lane == 0 && j < total) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a + 8u * buf), "r"(8192u) : "memory");
#pragma unroll
                for (uint32_t t = 0; t < kUnitTiles; ++t)
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(a_base + buf * 8192u + t * a_tile_bytes), "l"(&x_map),
                                   "r"(((j * kUnitTiles + t) % tiles_per_step) * 64u), "r"(0u), "r"(bar_a + 8u * buf)
                                 : "memory");
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        // ---- the issuing warp: one lane waits for a group's rows and, unit by unit, for x, and issues the matrix instructions ----
        uint32_t q = 0;
        for (uint32_t s = 0; s < P.steps; ++s) {
            const uint32_t acc = tmem + 32u * (s & 1u);
            for (uint32_t g = 0; g < P.groups; ++g, ++q) {
                if (lane == 0) {
                    bool ready = mbar_wait(bar_b + 8u * (q & 1u), (q >> 1) & 1u, abort_addr);
                    fence_async_smem();      // the rows' stores, ordered before this by the mbarrier, are read through the async proxy
                    // descriptors differ in their address field only: low word + (bytes >> 4)
                    const uint64_t da = umma_desc(a_base), db = umma_desc(b_base + G::kSlab * (q & 1u));
                    const uint32_t da_hi = uint32_t(da >> 32), db_hi = uint32_t(db >> 32), da_lo = uint32_t(da), db_lo = uint32_t(db);
#pragma unroll
                    for (uint32_t h = 0; h < kUnitsPerGroup; ++h) {
                        const uint32_t j = kUnitsPerGroup * q + h, buf = j & units_mask;
                        ready = ready && mbar_wait(bar_a + 8u * buf, (j >> depth) & 1u, abort_addr);
                        tc_fence_after();
#pragma unroll
                        for (uint32_t t = 0; t < kUnitTiles; ++t)
#pragma unroll
                            for (uint32_t k = 0; k < 4; ++k)             // 16 columns = 32 bytes further along the swizzled rows
                                if (ready)                               // (operands that never arrived are not multiplied)
                                    umma_bf16(acc, pack64(da_lo + ((buf * 8192u + t * a_tile_bytes + 32u * k) >> 4), da_hi),
                                              pack64(db_lo + (((h * kUnitTiles + t) * G::kBTile + 32u * k) >> 4), db_hi), G::kIdesc,
                                              (g | h | t | k) ? 1u : 0u);
                        umma_commit(bar_afree + 8u * buf);
                    }
                    umma_commit(bar_mma + 8u * (q & 1u));
                }
                __syncwarp();
            }
            if (TPAD > 16u) {                // tokens 16 .. are in this warp's quarter
                if (lane == 0) mbar_wait(bar_mma + 8u * ((q - 1u) & 1u), ((q - 1u) >> 1) & 1u, abort_addr);
                __syncwarp();
                read_out(s, 1u);
            }
        }
    } else if (warp < 2u + P.rows_per_step) {
        // ---- the decoding warps: one row of W each, group by group into the slabs of B ----
        const uint32_t w = warp - 2u, lt = (1u << lane) - 1u, ring = lut_addr + kRingBase + w * G::kRingStride, ctx = lut_addr + kCtxBase + w * kCtxBytes;
        const uint32_t k0 = __float_as_uint(float(4096 - J.zlo));
        const uint64_t kk = pack64(k0, k0);
        // where this lane's block of a group goes in a slab: 64-column tile lane / 8, row = w, piece lane % 8 of the row
        const uint32_t b_dst = b_base + (lane >> 3) * G::kBTile + w * 128u + (((lane & 7u) ^ (w & 7u)) << 4);
        // A row's record and scale are read a step ahead, so that a step begins with one read - its payload's - and not with two in a row
        // (10240 x 3840 at 4 bpp, 16 tokens, three steps of 15 groups: 51.1 -> 50.3 us; 24 rows of
        // 2048 columns at 3 bpp 12.3 -> 11.95).
        struct { uint32_t x, off, end, sigma; } next;
        auto ask = [&](uint32_t r) {
            const uint32_t tile = min(r, P.R - 1u);                     // = the row of W
            const uint32_t *rec = J.tile_index + size_t(tile) * 33u;
            next = {__ldg(rec + lane), __ldg(rec + 32), __ldg(rec + (tile + 1u < J.n_tiles ? 65u : 33u)), __float_as_uint(__ldg(J.scales + tile))};
        };
        ask(row_begin + w);
        uint32_t q = 0;
        for (uint32_t s = 0; s < P.steps; ++s) {
            const uint32_t r = row_begin + s * P.rows_per_step + w, act = r < row_end ? 1u : 0u;   // a CTA's last step may be short
            const TileSetup Tl = tile_setup(J, next.x, next.off, next.end);
            const uint32_t sigma = next.sigma;
            for (uint32_t c = 0; c < G::kSlots; ++c) ring_issue<G::kChunk, G::kSlots>(ring, Tl.a0, Tl.room, c, lane);
            const bool has_next = r + P.rows_per_step < row_end;
            ask(r + P.rows_per_step);
            if (lane == 0) {                 // the next request is chunk kSlots, into slot 0
                sts64(ctx + kCtxChain + kCcSrc, Tl.a0 + G::kRing);
                sts32(ctx + kCtxChain + kCcRem, Tl.room - G::kRing);
                sts32(ctx + kCtxChain + kCcDst, ring);
                sts32(ctx + kCtxChain + kCcRing, ring);
                sts32(ctx + kCtxChain + kCcWbase, ring);
            }
            cp_async_wait<1>();
            __syncwarp();
            if (has_next) {                  // the start of the next row's payload, into L2: 4 KB, the ring's first fill and more
                const uint64_t at = 2ull * min(next.off, J.total_words) + 128u * lane;
                if (at < 2ull * J.total_words) prefetch_l2(J.stream + J.off_payload + at);
            }
            uint32_t x = Tl.x, bal = 0, a = ring + Tl.lead;
            if (s == 0) wait_for_tables(tables);
            // The loop with fewer instructions (EP_BODY11); with the shorter chain of EP_BODY11_SHORT, one instruction more per step, us:
            //   16 tokens: 10240 x 3840 50.34 (this one 50.25), 4096 x 4096 22.80 (22.48), 8192 x 8192 79.7 (78.4), 60 rows per SM of 2560 columns
            //   29.14 (28.75), 4 rows of 4096 14.91 (15.02), 31 rows at 5 bpp 31.62 (31.81);
            //   32 tokens: 24 rows per SM of 4096 columns 24.96 (24.30), 70 rows 65.29 (63.08).
            EP_GEMM_ROW_ASM(EP_BODY11);
            cp_async_wait<0>();              // nothing may still be landing in the ring when the next row starts
            __syncwarp();
            const uint32_t pos = __shfl_sync(0xFFFFFFFFu, a, 0) + 2u * __popc(bal) - lds32(ctx + kCtxChain + kCcWbase);
            bad |= act && ((x != ep::kStateLow) || (Tl.off + ((pos - Tl.lead) >> 1) != Tl.end));
            __syncwarp();                    // the context block is rewritten for the next row
        }
    }
    const bool aborted = lds32(abort_addr) != 0;
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&g_ep_status, 1u);
    if (aborted && tid == 0) atomicOr(&g_ep_status, 2u);
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(64u) : "memory");
}

// ======================================================================================================
// Large-table path: b >= 12, a coordinate range above 1024, or a single-symbol table at b = 11.  The
// seventeen tables (2^b slots of 4 bytes: symbol index << 16 | u - F) are built into caller-provided
// scratch by one launch and read through L1/L2 by the decode launch that follows on the same stream; a
// symbol's frequency comes from the stream's own frequency arrays (a few KB, resident in L1) and its value
// is the table's minimum plus the index.  Slots are hit uniformly at random, so the traffic between L2 and
// L1 is what bounds this path: four-byte entries halve the table set (278 KB at b = 12, most of it
// L1-resident).  Same tile / lane / word order as above; payload words are read straight from global
// memory with the index clamped to the payload.
// ======================================================================================================

struct GJobParams {
    const uint8_t *stream;
    const uint32_t *tile_index;
    const float *scales;
    void *out;
    uint32_t *lut;                // scratch: 17 << b entries
    uint32_t off_tables;          // byte offset of the table section (directory, then frequencies)
    uint32_t off_payload;
    uint32_t total_words;
    uint32_t n_vec;
    uint32_t per_row;
    uint32_t V, n_tiles, b;
    uint32_t tile0, tile_cnt;     // the tiles this launch decodes
    uint32_t cta_begin, cta_count;
    // table geometry from the host's ep_info, never from the device copy of the directory
    int32_t tmin[EP_NUM_TABLES];
    uint16_t tK[EP_NUM_TABLES];
    uint32_t foff[EP_NUM_TABLES]; // start of table t's frequencies, in u16 units
    // two-level tables of a 2^12-slot stream (ep_build_tables12_kernel only)
    uint16_t *image;              // 16 x 4096 slots: twice the coordinate code
    uint32_t *hot;                // 16 x kHotSpan entries: the codes hs .. hs + kHotSpan - 1
    uint32_t *cold;               // 16 x kColdCodes entries: every code
    int32_t zlo;                  // coordinate value of code 0 (even)
    uint32_t hs;                  // first code of the hot window
};

struct GBatchParams {
    GJobParams job[EP_MAX_BATCH];
    int32_t n_jobs;
};

constexpr int kGThreads = 256;
constexpr int kGWarps = kGThreads / 32;

// exclusive prefix sum over the 1024 threads of a CTA (one thread adding the 1024 parts up took 13 us of a table build)
__device__ __forceinline__ uint32_t cta_exclusive_1024(uint32_t v, uint32_t *part) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= uint32_t(d)) incl += n;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    uint32_t w = part[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, w, d);
        if (lane >= uint32_t(d)) w += n;
    }
    const uint32_t before = __shfl_sync(0xFFFFFFFFu, w, int(warp) - 1 < 0 ? 0 : int(warp) - 1);
    return (warp ? before : 0u) + incl - v;
}

// one CTA per (table, job): exclusive prefix sums of the frequencies in shared memory (as u16; the last
// entry 2^b <= 32768 still fits), then every slot finds its symbol by binary search.  A table without symbols
// (or whose frequencies fall short of 2^b in a damaged stream) gets index 0 with offset 0 in the slots nobody owns.
__global__ void __launch_bounds__(1024) ep_build_tables_kernel(const __grid_constant__ GBatchParams P) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t part[32];
    const GJobParams &J = P.job[blockIdx.y];
    const uint32_t t = blockIdx.x, tid = threadIdx.x;
    const uint32_t K = J.tK[t];
    const uint32_t M = 1u << J.b;
    uint32_t *lut = J.lut + (size_t(t) << J.b);
    if (K == 0) {
        for (uint32_t u = tid; u < M; u += blockDim.x) lut[u] = 0u;
        return;
    }
    const uint16_t *fq = reinterpret_cast<const uint16_t *>(J.stream + J.off_tables + 8 * EP_NUM_TABLES) + J.foff[t];
    uint16_t *F = reinterpret_cast<uint16_t *>(smem);              // K + 1 entries
    const uint32_t per = (K + blockDim.x - 1) / blockDim.x;
    const uint32_t j0 = min(tid * per, K), j1 = min(j0 + per, K);
    uint32_t sum = 0;
    for (uint32_t j = j0; j < j1; ++j) sum += fq[j];
    uint32_t run = cta_exclusive_1024(sum, part);
    if (tid == 1023u) F[K] = uint16_t(min(run + sum, M));            // = 2^b for a valid stream
    for (uint32_t j = j0; j < j1; ++j) { F[j] = uint16_t(min(run, M)); run += fq[j]; }
    __syncthreads();
    for (uint32_t u = tid; u < M; u += blockDim.x) {
        uint32_t lo = 0, hi = K;                                     // largest j with F[j] <= u (F[0] = 0)
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (uint32_t(F[mid]) <= u) lo = mid; else hi = mid;
        }
        lut[u] = (lo << 16) | ((u - uint32_t(F[lo])) & 0xFFFFu);     // lo < K <= 65535
    }
}

// Two-level tables of a 2^12-slot stream (see EP_N1): one CTA per (coordinate table, job).  Prefix sums of the
// frequencies as above; then every code of the coordinate range gets its entry f << 16 | F in the complete array -
// and in the hot part, if it lies in the window of kHotSpan codes that the decode kernel keeps in shared memory -,
// and every slot finds its symbol by binary search and stores twice the symbol's code.  A code no symbol of the
// table has, and a symbol that never occurs, get f = 1 (they own no slot; the floor only keeps a damaged stream
// from producing states that take a word in every step).
__global__ void __launch_bounds__(1024) ep_build_tables12_kernel(const __grid_constant__ GBatchParams P) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t part[32];
    const GJobParams &J = P.job[blockIdx.y];
    const uint32_t t = blockIdx.x + 1u, tid = threadIdx.x;
    const uint32_t K = J.tK[t];
    constexpr uint32_t M = 4096;
    uint16_t *image = J.image + size_t(t - 1u) * M;
    uint32_t *hot = J.hot + (t - 1u) * kHotSpan;
    uint32_t *cold = J.cold + (t - 1u) * kColdCodes;
    const uint32_t unused = 1u << 16;                                 // f = 1, F = 0
    const bool is_m = ((t - 1u) & 7u) == 7u;                          // the m field: its coordinate is 2m (+ parity)
    if (K == 0) {
        for (uint32_t c = tid; c < kColdCodes; c += blockDim.x) cold[c] = unused;
        for (uint32_t c = tid; c < kHotSpan; c += blockDim.x) hot[c] = unused;
        for (uint32_t u = tid; u < M; u += blockDim.x) image[u] = 0;  // never looked up in a valid stream
        return;
    }
    const uint16_t *fq = reinterpret_cast<const uint16_t *>(J.stream + J.off_tables + 8 * EP_NUM_TABLES) + J.foff[t];
    uint16_t *F = reinterpret_cast<uint16_t *>(smem);              // K + 1 entries
    const uint32_t per = (K + blockDim.x - 1) / blockDim.x;
    const uint32_t j0 = min(tid * per, K), j1 = min(j0 + per, K);
    uint32_t sum = 0;
    for (uint32_t j = j0; j < j1; ++j) sum += fq[j];
    uint32_t run = cta_exclusive_1024(sum, part);
    if (tid == 1023u) F[K] = uint16_t(min(run + sum, M));
    for (uint32_t j = j0; j < j1; ++j) { F[j] = uint16_t(min(run, M)); run += fq[j]; }
    __syncthreads();
    for (uint32_t c = tid; c < kColdCodes; c += blockDim.x) {
        const int32_t z = int32_t(c) + J.zlo;                         // the coordinate value of this code
        const int32_t j = (is_m ? (z >> 1) : z) - J.tmin[t];          // (z even for the m field: the shift is exact)
        uint32_t e = unused;
        if (!(is_m && (z & 1)) && j >= 0 && uint32_t(j) < K)
            e = (min(max(uint32_t(fq[j]), 1u), M) << 16) | min(uint32_t(F[j]), M - 1u);
        cold[c] = e;
        if (c - J.hs < kHotSpan) hot[c - J.hs] = e;                   // (unsigned: a code below the window wraps)
    }
    for (uint32_t u = tid; u < M; u += blockDim.x) {
        uint32_t lo = 0, hi = K;                                     // largest j with F[j] <= u (F[0] = 0)
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (uint32_t(F[mid]) <= u) lo = mid; else hi = mid;
        }
        const int32_t z = J.tmin[t] + int32_t(lo);
        const int32_t code = (is_m ? 2 * z : z) - J.zlo;
        image[u] = uint16_t(2 * min(max(code, 0), int32_t(kColdCodes) - 1));
    }
}

// one symbol: returns its index inside table t's symbol range (0 for an idle lane); Kmax = the table's last index
__device__ __forceinline__ uint32_t grans_step(uint32_t &x, const uint32_t *table, const uint16_t *freq, uint32_t Kmax,
                                               uint32_t mask, uint32_t b, uint32_t &ptr, const uint16_t *pay, uint32_t lt,
                                               bool act, uint32_t last_word) {
    uint32_t sym = 0;
    bool need = false;
    if (act) {
        const uint32_t e = __ldg(table + (x & mask));
        sym = min(e >> 16, Kmax);                 // whatever the scratch holds, stay inside the frequency array
        x = uint32_t(__ldg(freq + sym)) * (x >> b) + (e & 0xFFFFu);
        need = x < ep::kStateLow;
    }
    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, need);
    if (need) x = (x << 16) | __ldg(pay + min(ptr + __popc(bal & lt), last_word));
    ptr += __popc(bal);
    return sym;
}

template <int DT>
__global__ void __launch_bounds__(kGThreads) ep_decode_glut_kernel(const __grid_constant__ GBatchParams P) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    int j = 0;
    while (j + 1 < P.n_jobs && blockIdx.x >= P.job[j + 1].cta_begin) ++j;
    const GJobParams &J = P.job[j];
    const uint16_t *fq = reinterpret_cast<const uint16_t *>(J.stream + J.off_tables + 8 * EP_NUM_TABLES);
    const uint32_t b = J.b, mask = (1u << b) - 1u, lt = (1u << lane) - 1u;
    const uint16_t *pay = reinterpret_cast<const uint16_t *>(J.stream + J.off_payload);
    const uint32_t last_word = J.total_words ? J.total_words - 1u : 0u;
    const uint32_t cta = blockIdx.x - J.cta_begin;
    const uint32_t K0max = J.tK[0] ? J.tK[0] - 1u : 0u;
    for (uint32_t local = cta * kGWarps + warp; local < J.tile_cnt; local += J.cta_count * kGWarps) {
        const uint32_t tile = J.tile0 + local;
        const uint32_t *rec = J.tile_index + size_t(tile) * 33u;
        uint32_t x = rec[lane];
        uint32_t ptr = rec[32];
        const uint32_t end = (tile + 1 < J.n_tiles) ? rec[33 + 32] : rec[33];
        const uint32_t v0 = tile * J.V;
        const uint32_t nv = min(J.V, J.n_vec - v0);
        for (uint32_t g = 0; g * 32u < nv; ++g) {
            const uint32_t i = g * 32u + lane;
            const bool act = i < nv;
            int32_t fld[9];
            fld[0] = int32_t(grans_step(x, J.lut, fq + J.foff[0], K0max, mask, b, ptr, pay, lt, act, last_word)) + J.tmin[0];
            const uint32_t t0 = 1u + 8u * uint32_t(fld[0] & 1);          // first coordinate table of this coset
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k) {
                const uint32_t t = t0 + k;
                const uint32_t Kt = J.tK[t];
                fld[k + 1] = int32_t(grans_step(x, J.lut + (size_t(t) << b), fq + J.foff[t], Kt ? Kt - 1u : 0u, mask, b, ptr, pay,
                                                lt, act && Kt != 0u, last_word)) + J.tmin[t];
            }
            if (!act) continue;
            const uint32_t v = v0 + i;
            if constexpr (DT == EP_FIELDS_I32) {
                int32_t *o = static_cast<int32_t *>(J.out) + size_t(v) * 9u;
#pragma unroll
                for (int k = 0; k < 9; ++k) o[k] = fld[k];
            } else {
                // Eq. 5 on doubled coordinates q = 2p (integers), then p = q/2 exactly and Eq. 19
                const float sigma = __ldg(J.scales + v / J.per_row);
                int32_t s7 = 0;
                float w[8];
#pragma unroll
                for (int k = 1; k <= 7; ++k) {
                    s7 += fld[k];
                    w[k - 1] = __fmul_rn(sigma, float(2 * fld[k] + fld[0]) * 0.5f);
                }
                w[7] = __fmul_rn(sigma, float(2 * (2 * fld[8] + (s7 & 1)) + fld[0]) * 0.5f);
                Out<DT>::store(static_cast<uint8_t *>(J.out) + size_t(v) * Out<DT>::kBlockBytes, w);
            }
        }
        const bool bad = (x != ep::kStateLow) || (ptr != end);
        if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicOr(&g_ep_status, 1u);
    }
}

// A prepared image of the sixteen shared-memory tables in global memory (ep_prepare_tables): one CTA per table.  Prefix sums of
// the frequencies, then every slot finds its symbol by binary search; the entries are build_one_table's.  (One CTA with
// a warp per table, as in the decode kernel, took 8.4 us, most of it the serial loop over the symbols of many slots.)
constexpr uint32_t kPrepThreads = 256, kPrepPer = kLutEntries / kPrepThreads;
__global__ void __launch_bounds__(kPrepThreads) ep_prepare_tables_kernel(const __grid_constant__ JobParams J, uint32_t *image) {
    __shared__ uint32_t first[kLutEntries + 1], part[kPrepThreads / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, t = 1u + blockIdx.x, K = J.tK[t];      // K <= 2048 (see fits_smem_tables)
    wait_for_stream();
    const uint16_t *fq = reinterpret_cast<const uint16_t *>(J.stream + J.off_freq) + J.foff[t];
    uint32_t f[kPrepPer], sum = 0;
#pragma unroll
    for (uint32_t i = 0; i < kPrepPer; ++i) {
        const uint32_t j = tid * kPrepPer + i;
        f[i] = j < K ? uint32_t(fq[j]) : 0u;
        if (f[i] >= kLutEntries) atomicOr(&g_ep_status, 1u);
        sum += f[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= uint32_t(d)) incl += n;
    }
    if (lane == 31) part[tid >> 5] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
    for (uint32_t w = 0; w < tid >> 5; ++w) run += part[w];
#pragma unroll
    for (uint32_t i = 0; i < kPrepPer; ++i) {
        if (tid * kPrepPer + i <= K) first[tid * kPrepPer + i] = run;
        run += f[i];
    }
    if (tid == kPrepThreads - 1u && K == kLutEntries) first[K] = run;
    __syncthreads();
    const uint32_t total = first[K], slots = 1u << J.b;
    const bool is_m = ((t - 1u) & 7u) == 7u;
    for (uint32_t u = tid; u < kLutEntries; u += kPrepThreads) {
        uint32_t e = kEntryUnused;                       // slots no symbol owns (a damaged stream) or that b < 11 does not have
        if (u < min(total, slots)) {
            uint32_t lo = 0, hi = K;                     // largest j with first[j] <= u
            while (hi - lo > 1u) {
                const uint32_t mid = (lo + hi) >> 1;
                if (first[mid] <= u) lo = mid; else hi = mid;
            }
            const int32_t v = J.tmin[t] + int32_t(lo);
            const uint32_t code = uint32_t((is_m ? 2 * v : v) - J.zlo);
            e = (min(first[lo + 1u] - first[lo], kLutEntries - 1u) << 21) | ((code & 0x3FFu) << 11) | (u - first[lo]);
        }
        image[(t - 1u) * kLutEntries + u] = e;
    }
}

// ---- host side -----------------------------------------------------------------------------------

// the tiles a job asks for: its range, or the whole tensor when both range fields are 0
inline uint32_t job_tile0(const ep_decode_job &jb) { return jb.tile_count ? jb.tile_begin : 0u; }
inline uint32_t job_tiles(const ep_decode_job &jb) { return jb.tile_count ? jb.tile_count : jb.info->n_tiles; }

int g_num_sms[64] = {};

int num_sms() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64 && g_num_sms[dev]) return g_num_sms[dev];
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64) g_num_sms[dev] = n;
    return n;
}

struct Range { int64_t lo, hi; bool any; };

// coordinate range from the table directory (the header's coord_min/max are not trusted)
Range coord_range(const ep_info &I) {
    Range r{0, 0, false};
    for (int c = 0; c < 2; ++c)
        for (int k = 1; k <= 8; ++k) {
            const int t = ep::table_id(c, k);
            if (!I.table_K[t]) continue;
            int64_t lo = I.table_min[t], hi = int64_t(I.table_min[t]) + I.table_K[t] - 1;
            if (k == 8) { lo *= 2; hi = 2 * hi + 1; }
            if (!r.any) { r = {lo, hi, true}; }
            else { r.lo = lo < r.lo ? lo : r.lo; r.hi = hi > r.hi ? hi : r.hi; }
        }
    return r;
}

int64_t even_base(const Range &r) {
    int64_t zlo = r.any ? r.lo : 0;
    if (zlo > -2) zlo = -2;
    return zlo & ~int64_t(1);   // floor to even
}

bool fits_smem_tables(const ep_info &I) {
    if (I.b > 11) return false;
    const Range r = coord_range(I);
    const int64_t zlo = even_base(r);
    if (r.any && r.hi - zlo > 1023) return false;     // 10-bit code field
    if (zlo < -1024) return false;                    // 4096 - zlo stays below 8192: same fp32 exponent as 4096 + code
    for (int t = 1; t < EP_NUM_TABLES; ++t) {         // (the coset table is decoded by comparison: any frequency goes)
        if (I.table_K[t] > kLutEntries) return false;
        if (I.b == 11 && I.table_K[t] == 1) return false;   // a lone symbol has f = 2^11: one bit more than the f field
    }
    return true;
}

// table geometry of a job whose tables fit shared memory
void fill_table_params(JobParams &J, const ep_info &I) {
    J.off_freq = I.off_tables + 8u * EP_NUM_TABLES;
    J.b = I.b;
    J.zlo = int32_t(even_base(coord_range(I)));
    uint32_t acc = 0;
    for (int t = 0; t < EP_NUM_TABLES; ++t) {
        J.tmin[t] = int16_t(I.table_min[t]);
        J.tK[t] = uint16_t(I.table_K[t]);
        J.foff[t] = uint16_t(acc);
        acc += I.table_K[t];
    }
}

// A launch that may overlap the end of the kernel before it (see wait_for_stream, which `kernel` begins with): the next
// decode is then resident when its turn comes instead of being launched then.
template <class... A>
cudaError_t launch_next(void (*kernel)(A...), uint32_t grid, uint32_t threads, uint32_t smem, cudaStream_t st, const A &...args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// How the tiles of a launch are spread over its CTAs (persistent, one per SM): sets tiles_per_round, every job's rounds and
// costs and cost_per_cta; returns the grid size, 0 if the counts do not fit 32 bits.
// A round is one tile per warp, and its warps share an SM's issue slots: 32 of them take 1.05 us for a group of 32 blocks
// each, 8 take 0.7.  So the fewest rounds per CTA that 32 tiles at a time allow are kept, and then a round gets no more
// tiles than it takes to spread them over all SMs in that many rounds: a 4096 x 4096 tensor of 1152 tiles runs as 144
// CTAs of eight warps, not as 36 of 32.  With one round per CTA every CTA simply takes one; with more, the
// cost-weighted list of all rounds is split evenly.
uint32_t split_rounds(BatchParams &P, uint32_t sms) {
    auto rounds_at = [&](uint32_t tpr) {
        uint64_t n = 0;
        for (int i = 0; i < P.n_jobs; ++i) n += (uint64_t(P.job[i].tile_cnt) + tpr - 1u) / tpr;
        return n;
    };
    const uint64_t most = (rounds_at(kTilesPerRound) + sms - 1u) / sms * sms;
    uint32_t lo = 1, hi = kTilesPerRound;                      // smallest tiles_per_round with at most `most` rounds
    while (lo < hi) {
        const uint32_t mid = (lo + hi) / 2u;
        if (rounds_at(mid) <= most) hi = mid; else lo = mid + 1u;
    }
    P.tiles_per_round = lo;
    const uint64_t rounds_total = rounds_at(lo);
    uint64_t cost = 0;
    for (int i = 0; i < P.n_jobs; ++i) {
        JobParams &J = P.job[i];
        J.rounds = (J.tile_cnt + lo - 1u) / lo;
        J.round_cost = rounds_total <= sms ? 1u : (J.V + 31u) / 32u;
        J.cost_begin = uint32_t(cost);
        cost += uint64_t(J.rounds) * J.round_cost;
        uint32_t tables = 0, symbols = 0;                    // of the coordinates
        for (int t = 1; t < EP_NUM_TABLES; ++t) { tables += J.tK[t] != 0; symbols += J.tK[t]; }
        J.guess = tables && ep::guess_pays(lo, J.V < J.n_vec ? J.V : J.n_vec, J.payload_bits, double(symbols) / tables);
    }
    const uint32_t grid = uint32_t(rounds_total < sms ? rounds_total : sms);
    // (a tensor has under 2^27 blocks, so sixteen of them cost under 2^28 groups and rounds: 32-bit arithmetic in the kernel)
    if (cost + grid >= (1ull << 31)) return 0;
    P.cost_per_cta = uint32_t((cost + grid - 1u) / grid);
    return grid;
}

template <int DT, bool FEW>
cudaError_t launch_smem_as(const BatchParams &P, uint32_t grid, uint32_t warps, cudaStream_t st) {
    static bool configured[64] = {};   // the attribute is per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(ep_decode_smem_kernel<DT, FEW>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes));
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    uint32_t least = kMinWarps;
    for (int i = 0; i < P.n_jobs; ++i)
        if (!P.job[i].lut_image) least = kBuildWarps;
    return launch_next(ep_decode_smem_kernel<DT, FEW>, grid, 32u * (warps < least ? least : warps), kSmemBytes, st, P);
}
template <int DT>
cudaError_t launch_smem(const BatchParams &P, uint32_t grid, cudaStream_t st) {
    const uint32_t warps = P.tiles_per_round;
    bool few = warps <= kFewTiles;
    for (int i = 0; i < P.n_jobs && few; ++i)        // room for a tile's row scales and a window of 4 KB
        few = 4u * (uint64_t(P.job[i].V) / P.job[i].per_row + 3u) + 128u + 4096u <= kStageBytes / warps;
    return few ? launch_smem_as<DT, true>(P, grid, warps, st) : launch_smem_as<DT, false>(P, grid, warps, st);
}

size_t large_table_bytes(const ep_info &I) { return size_t(EP_NUM_TABLES) * (size_t(1) << I.b) * 4u; }

// 2^12-slot streams whose coordinates span at most kColdCodes values decode from two-level tables in the hot loop
bool fits_two_level(const ep_info &I) {
    if (I.b != 12) return false;
    const Range r = coord_range(I);
    const int64_t zlo = even_base(r);
    return r.any && r.hi - zlo < int64_t(kColdCodes) && zlo >= -(int64_t(1) << 20);   // 2^22 - zlo and 2^22 + code: one exponent
}
// first code of the hot window: kHotSpan codes centred on the coordinate value 0, kept inside the code range
uint32_t hot_start(const ep_info &I) {
    const Range r = coord_range(I);
    const int64_t zlo = even_base(r), codes = (r.any ? r.hi : 0) - zlo + 1;
    const int64_t last = codes > int64_t(kHotSpan) ? codes - int64_t(kHotSpan) : 0;
    int64_t hs = -zlo - int64_t(kHotSpan / 2);
    if (hs < 0) hs = 0;
    return uint32_t(hs < last ? hs : last);
}
// image, hot part, complete array; the flat tables of the large-table kernel follow at this offset
size_t two_level_bytes(const ep_info &) { return size_t(kLutBytes) + kHotBytes + kColdBytes; }
// can the hot loop serve this request?  (the field dump and narrow tensors take the plain kernels)
bool hot_loop_shape(const ep_info &I, int32_t dt) { return dt != EP_FIELDS_I32 && I.C / 8 >= 32u && I.V < (1u << 20); }

// the host-side parameters of a large-table job (geometry from `info` only); `lut` = where its tables are or go
int fill_large_job(GJobParams &J, const ep_decode_job &jb, uint32_t *lut) {
    const ep_info &I = *jb.info;
    uint32_t acc = 0;
    for (int t = 0; t < EP_NUM_TABLES; ++t) {
        if (I.table_K[t] > 65535u) return EP_ERR_UNSUPPORTED;
        J.tmin[t] = I.table_min[t];
        J.tK[t] = uint16_t(I.table_K[t]);
        J.foff[t] = acc;
        acc += I.table_K[t];
    }
    J.stream = static_cast<const uint8_t *>(jb.d_stream);
    J.tile_index = static_cast<const uint32_t *>(jb.d_tile_index);
    J.scales = jb.d_row_scales;
    J.out = jb.d_out;
    J.lut = lut;
    J.off_tables = I.off_tables;
    J.off_payload = I.off_payload;
    J.total_words = uint32_t(I.total_words);
    J.n_vec = uint32_t(uint64_t(I.R) * (I.C / 8));
    J.per_row = I.C / 8;
    J.V = I.V;
    J.n_tiles = I.n_tiles;
    J.b = I.b;
    return EP_OK;
}

// where the two-level tables of a job live inside its table buffer
void set_two_level(GJobParams &J, const ep_info &I, void *base) {
    J.image = static_cast<uint16_t *>(base);
    J.hot = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(base) + kLutBytes);
    J.cold = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(base) + kLutBytes + kHotBytes);
    J.zlo = int32_t(even_base(coord_range(I)));
    J.hs = hot_start(I);
}

cudaError_t launch_build12(const GBatchParams &P, int n_jobs, cudaStream_t st) {
    uint32_t max_K = 1;
    for (int i = 0; i < n_jobs; ++i)
        for (int t = 1; t < EP_NUM_TABLES; ++t)
            if (P.job[i].tK[t] > max_K) max_K = P.job[i].tK[t];
    const size_t smem = 2u * (size_t(max_K) + 1u);
    if (smem > 48u * 1024u) {
        const cudaError_t e = cudaFuncSetAttribute(ep_build_tables12_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    ep_build_tables12_kernel<<<dim3(EP_NUM_TABLES - 1, n_jobs), 1024, smem, st>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_build(const GBatchParams &P, int n_jobs, cudaStream_t st) {
    uint32_t max_K = 1;
    for (int i = 0; i < n_jobs; ++i)
        for (int t = 0; t < EP_NUM_TABLES; ++t)
            if (P.job[i].tK[t] > max_K) max_K = P.job[i].tK[t];
    const size_t smem = 2u * (size_t(max_K) + 1u);
    if (smem > 48u * 1024u) {
        const cudaError_t e = cudaFuncSetAttribute(ep_build_tables_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    ep_build_tables_kernel<<<dim3(EP_NUM_TABLES, n_jobs), 1024, smem, st>>>(P);
    return cudaGetLastError();
}

}  // namespace

extern "C" size_t ep_decode_scratch_bytes(const ep_info *info) {
    if (!info) return 0;
    if (fits_smem_tables(*info)) return 0;
    return (fits_two_level(*info) ? two_level_bytes(*info) : 0) + large_table_bytes(*info);
}

extern "C" size_t ep_decode_tables_bytes(const ep_info *info) {
    if (!info) return 0;
    return fits_smem_tables(*info) ? size_t(kLutBytes) : ep_decode_scratch_bytes(info);
}

extern "C" uint32_t ep_decode_tiles_per_sm(void) { return kTilesPerRound; }

extern "C" int ep_prepare_tables(const ep_info *info, const void *d_stream, void *d_tables, size_t tables_bytes, void *stream) {
    if (!info || !d_stream || !d_tables) return EP_ERR_BAD_ARG;
    const ep_info &I = *info;
    if (I.b < 9 || I.b > 15 || (reinterpret_cast<uintptr_t>(d_stream) & 3)) return EP_ERR_BAD_ARG;
    if (tables_bytes < ep_decode_tables_bytes(info) || (reinterpret_cast<uintptr_t>(d_tables) & 255)) return EP_ERR_SCRATCH;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (fits_smem_tables(I)) {
        JobParams J;
        std::memset(&J, 0, sizeof(J));
        J.stream = static_cast<const uint8_t *>(d_stream);
        fill_table_params(J, I);
        return launch_next(ep_prepare_tables_kernel, EP_NUM_TABLES - 1, kPrepThreads, 0, st, J, static_cast<uint32_t *>(d_tables)) == cudaSuccess
                   ? EP_OK : EP_ERR_CUDA;
    }
    GBatchParams P;
    std::memset(&P, 0, sizeof(P));
    P.n_jobs = 1;
    ep_decode_job jb;
    std::memset(&jb, 0, sizeof(jb));
    jb.info = info;
    jb.d_stream = d_stream;
    // a 2^12-slot stream gets the two-level tables of the hot loop first, then the flat tables the plain kernel
    // uses for the field dump and for narrow tensors
    uint8_t *base = static_cast<uint8_t *>(d_tables);
    const bool two = fits_two_level(I);
    const int rc = fill_large_job(P.job[0], jb, reinterpret_cast<uint32_t *>(base + (two ? two_level_bytes(I) : 0)));
    if (rc) return rc;
    if (two) {
        set_two_level(P.job[0], I, base);
        if (launch_build12(P, 1, st) != cudaSuccess) return EP_ERR_CUDA;
    }
    return launch_build(P, 1, st) == cudaSuccess ? EP_OK : EP_ERR_CUDA;
}

namespace {

template <int DT>
cudaError_t launch_glut(const GBatchParams &P, uint32_t grid, cudaStream_t st) {
    ep_decode_glut_kernel<DT><<<grid, kGThreads, 0, st>>>(P);
    return cudaGetLastError();
}

// jobs whose tables do not fit shared memory: decode from tables in global memory - the caller's prepared
// ones, or tables built into the caller's scratch by one extra launch first
int decode_large_tables(const ep_decode_job *const *jobs, int n_jobs, int32_t dt, int sms, cudaStream_t st) {
    GBatchParams P, B;      // B: the jobs whose tables have to be built
    std::memset(&P, 0, sizeof(P));
    std::memset(&B, 0, sizeof(B));
    P.n_jobs = n_jobs;
    uint32_t next = 0;
    int n_build = 0;
    for (int i = 0; i < n_jobs; ++i) {
        const ep_decode_job &jb = *jobs[i];
        const ep_info &I = *jb.info;
        // the flat tables follow the two-level ones where the buffer has both (prepared tables always, scratch
        // if it is large enough); a scratch buffer of the flat tables' size alone holds just them
        const size_t need = large_table_bytes(I), before = fits_two_level(I) ? two_level_bytes(I) : 0;
        uint32_t *lut;
        if (jb.d_tables) {
            if (reinterpret_cast<uintptr_t>(jb.d_tables) & 255) return EP_ERR_SCRATCH;
            lut = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(const_cast<void *>(jb.d_tables)) + before);
        } else {
            if (!jb.d_scratch || jb.scratch_bytes < need || (reinterpret_cast<uintptr_t>(jb.d_scratch) & 255)) return EP_ERR_SCRATCH;
            lut = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(jb.d_scratch) + (jb.scratch_bytes >= before + need ? before : 0));
        }
        GJobParams &J = P.job[i];
        const int rc = fill_large_job(J, jb, lut);
        if (rc) return rc;
        J.tile0 = job_tile0(jb);
        J.tile_cnt = job_tiles(jb);
        const uint64_t want = (uint64_t(J.tile_cnt) + kGWarps - 1) / kGWarps;
        const uint64_t cap = uint64_t(sms) * 8u;
        J.cta_begin = next;
        J.cta_count = uint32_t(want < cap ? want : cap);
        next += J.cta_count;
        if (!jb.d_tables) B.job[n_build++] = J;
    }
    if (n_build) {
        B.n_jobs = n_build;
        if (launch_build(B, n_build, st) != cudaSuccess) return EP_ERR_CUDA;
    }
    cudaError_t e;
    switch (dt) {
    case EP_BF16: e = launch_glut<EP_BF16>(P, next, st); break;
    case EP_FP16: e = launch_glut<EP_FP16>(P, next, st); break;
    case EP_FP8_E4M3: e = launch_glut<EP_FP8_E4M3>(P, next, st); break;
    case EP_INT8: e = launch_glut<EP_INT8>(P, next, st); break;
    case EP_FP32: e = launch_glut<EP_FP32>(P, next, st); break;
    case EP_FP8_E5M2: e = launch_glut<EP_FP8_E5M2>(P, next, st); break;
    case EP_UINT8: e = launch_glut<EP_UINT8>(P, next, st); break;
    case EP_FIELDS_I32: e = launch_glut<EP_FIELDS_I32>(P, next, st); break;
    default: return EP_ERR_BAD_ARG;
    }
    return e == cudaSuccess ? EP_OK : EP_ERR_CUDA;
}

}  // namespace

extern "C" int ep_decode_batch(const ep_decode_job *jobs_in, int32_t n_in, void *stream) {
    if (!jobs_in || n_in <= 0 || n_in > EP_MAX_BATCH) return EP_ERR_BAD_ARG;
    const int sms = num_sms();
    if (sms <= 0) return EP_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int32_t dt = jobs_in[0].out_dtype;
    if (dt != EP_BF16 && dt != EP_FP16 && dt != EP_FP8_E4M3 && dt != EP_INT8 && dt != EP_FP32 && dt != EP_FP8_E5M2 &&
        dt != EP_UINT8 && dt != EP_FIELDS_I32)
        return EP_ERR_BAD_ARG;
    const ep_decode_job *fast[EP_MAX_BATCH], *large[EP_MAX_BATCH];
    int n_jobs = 0, n_large = 0;
    for (int i = 0; i < n_in; ++i) {
        const ep_decode_job &jb = jobs_in[i];
        if (!jb.info || !jb.d_stream || !jb.d_tile_index || !jb.d_out) return EP_ERR_BAD_ARG;
        if (jb.out_dtype != dt) return EP_ERR_BAD_ARG;   // one output type per launch
        if (dt != EP_FIELDS_I32 && !jb.d_row_scales) return EP_ERR_BAD_ARG;
        const ep_info &I = *jb.info;
        if (I.C == 0 || I.C % 8 || I.R == 0 || I.V == 0 || I.b < 9 || I.b > 15 || I.J != ep::kStates) return EP_ERR_BAD_ARG;
        // one vector store per block: 16 bytes for the two-byte types (two of them for FP32), 8 for the one-byte types
        const uintptr_t out_mask = dt == EP_FIELDS_I32 ? 3u : (dt == EP_FP8_E4M3 || dt == EP_FP8_E5M2 || dt == EP_INT8 || dt == EP_UINT8) ? 7u : 15u;
        if ((reinterpret_cast<uintptr_t>(jb.d_stream) & 3) || (reinterpret_cast<uintptr_t>(jb.d_tile_index) & 3) ||
            (reinterpret_cast<uintptr_t>(jb.d_out) & out_mask))
            return EP_ERR_BAD_ARG;
        if (I.table_K[0] == 0 || I.table_min[0] < 0 || int64_t(I.table_min[0]) + I.table_K[0] > 2) return EP_ERR_BAD_STREAM;
        // 32-bit byte offsets into the output (one row and one group beyond the end still representable) and a
        // signed 32-bit payload remainder in the kernels
        if ((uint64_t(I.R) + 1u) * I.C * 4u + 1024u >= (1ull << 32) || I.total_words >= (1ull << 30)) return EP_ERR_UNSUPPORTED;
        if (jb.tile_count != 0 || jb.tile_begin != 0) {     // a tile range: inside the tensor and not empty
            if (jb.tile_count == 0 || jb.tile_begin >= I.n_tiles || jb.tile_count > I.n_tiles - jb.tile_begin) return EP_ERR_BAD_ARG;
        }
        if (fits_smem_tables(I)) { fast[n_jobs++] = &jb; }
        else if (fits_two_level(I) && hot_loop_shape(I, dt) &&
                 (jb.d_tables || (jb.d_scratch && jb.scratch_bytes >= two_level_bytes(I)))) { fast[n_jobs++] = &jb; }
        else large[n_large++] = &jb;
    }
    if (n_large) {
        const int rc = decode_large_tables(large, n_large, dt, sms, st);
        if (rc) return rc;
    }
    if (n_jobs == 0) return EP_OK;
    BatchParams P;
    std::memset(&P, 0, sizeof(P));
    P.n_jobs = n_jobs;
    GBatchParams B12;               // two-level tables that have to be built into scratch first
    std::memset(&B12, 0, sizeof(B12));
    int n_build12 = 0;
    for (int i = 0; i < n_jobs; ++i) {
        const ep_decode_job &jb = *fast[i];
        const ep_info &I = *jb.info;
        JobParams &J = P.job[i];
        const uint32_t my_tiles = job_tiles(jb);
        if (jb.d_tables && (reinterpret_cast<uintptr_t>(jb.d_tables) & 255)) return EP_ERR_SCRATCH;
        J.stream = static_cast<const uint8_t *>(jb.d_stream);
        J.tile_index = static_cast<const uint32_t *>(jb.d_tile_index);
        J.scales = jb.d_row_scales;
        J.out = jb.d_out;
        J.lut_image = static_cast<const uint32_t *>(jb.d_tables);
        if (I.b == 12) {            // two-level tables: prepared, or built into the caller's scratch by a launch before this one
            void *base = const_cast<void *>(jb.d_tables);
            if (!base) {
                if (reinterpret_cast<uintptr_t>(jb.d_scratch) & 255) return EP_ERR_SCRATCH;
                base = jb.d_scratch;
                GJobParams &G = B12.job[n_build12++];
                const int rc = fill_large_job(G, jb, nullptr);
                if (rc) return rc;
                set_two_level(G, I, base);
            }
            J.lut_image = static_cast<const uint32_t *>(base);
            J.cold = reinterpret_cast<const uint32_t *>(static_cast<const uint8_t *>(base) + kLutBytes + kHotBytes);
            J.hs2 = 2u * hot_start(I);
        }
        J.off_payload = I.off_payload;
        J.total_words = uint32_t(I.total_words);
        J.n_vec = uint32_t(uint64_t(I.R) * (I.C / 8));
        J.per_row = I.C / 8;
        J.V = I.V;
        J.n_tiles = I.n_tiles;
        J.tile0 = job_tile0(jb);
        J.tile_cnt = my_tiles;
        fill_table_params(J, I);
        const uint32_t block_bytes = dt == EP_FIELDS_I32 ? 36u : dt == EP_FP32 ? 32u : (dt == EP_BF16 || dt == EP_FP16) ? 16u : 8u;
        J.row_bytes = J.per_row * block_bytes;
        J.row_rcp = uint32_t(0xFFFFFFFFu / J.row_bytes + 1u);
        J.row_max = I.R - 1u;
        J.payload_bits = float(double(I.total_words) * 16.0 / (9.0 * double(J.n_vec)));
    }
    const uint32_t next = split_rounds(P, uint32_t(sms));      // grid size
    if (next == 0) return EP_ERR_UNSUPPORTED;
    if (n_build12) {
        B12.n_jobs = n_build12;
        if (launch_build12(B12, n_build12, st) != cudaSuccess) return EP_ERR_CUDA;
    }
    cudaError_t e;
    switch (dt) {
    case EP_BF16: e = launch_smem<EP_BF16>(P, next, st); break;
    case EP_FP16: e = launch_smem<EP_FP16>(P, next, st); break;
    case EP_FP8_E4M3: e = launch_smem<EP_FP8_E4M3>(P, next, st); break;
    case EP_INT8: e = launch_smem<EP_INT8>(P, next, st); break;
    case EP_FP32: e = launch_smem<EP_FP32>(P, next, st); break;
    case EP_FP8_E5M2: e = launch_smem<EP_FP8_E5M2>(P, next, st); break;
    case EP_UINT8: e = launch_smem<EP_UINT8>(P, next, st); break;
    case EP_FIELDS_I32: e = launch_smem<EP_FIELDS_I32>(P, next, st); break;
    default: return EP_ERR_BAD_ARG;
    }
    return e == cudaSuccess ? EP_OK : EP_ERR_CUDA;
}

namespace {
ep_decode_job one_job(const ep_info *info, const void *d_stream, const void *d_tile_index, const float *d_row_scales,
                      int32_t out_dtype, void *d_out, void *d_scratch, size_t scratch_bytes) {
    ep_decode_job jb;
    std::memset(&jb, 0, sizeof(jb));
    jb.info = info;
    jb.d_stream = d_stream;
    jb.d_tile_index = d_tile_index;
    jb.d_row_scales = d_row_scales;
    jb.out_dtype = out_dtype;
    jb.d_out = d_out;
    jb.d_scratch = d_scratch;
    jb.scratch_bytes = scratch_bytes;
    return jb;
}
}  // namespace

extern "C" int ep_decode_tiles(const ep_info *info, const void *d_stream, const void *d_tile_index,
                               const float *d_row_scales, int32_t out_dtype, void *d_out, void *d_scratch,
                               size_t scratch_bytes, uint32_t tile_begin, uint32_t tile_count, void *stream) {
    if (tile_count == 0) return EP_ERR_BAD_ARG;
    ep_decode_job jb = one_job(info, d_stream, d_tile_index, d_row_scales, out_dtype, d_out, d_scratch, scratch_bytes);
    jb.tile_begin = tile_begin;
    jb.tile_count = tile_count;
    return ep_decode_batch(&jb, 1, stream);
}

extern "C" int ep_decode_tensor(const ep_info *info, const void *d_stream, const void *d_tile_index,
                                const float *d_row_scales, int32_t out_dtype, void *d_out, void *d_scratch,
                                size_t scratch_bytes, void *stream) {
    const ep_decode_job jb = one_job(info, d_stream, d_tile_index, d_row_scales, out_dtype, d_out, d_scratch, scratch_bytes);
    return ep_decode_batch(&jb, 1, stream);
}

namespace {
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                   const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
}

extern "C" int ep_decode_gemm(const ep_info *info, const void *d_stream, const void *d_tile_index, const float *d_row_scales,
                              const void *d_tables, const void *d_x, uint32_t T, float *d_y, void *stream) {
    if (!info || !d_stream || !d_tile_index || !d_row_scales || !d_tables || !d_x || !d_y || T == 0) return EP_ERR_BAD_ARG;
    const ep_info &I = *info;
    if (I.C == 0 || I.C % 8 || I.R == 0 || I.V == 0 || I.b < 9 || I.b > 15 || I.J != ep::kStates) return EP_ERR_BAD_ARG;
    if ((reinterpret_cast<uintptr_t>(d_stream) & 3) || (reinterpret_cast<uintptr_t>(d_tile_index) & 3) ||
        (reinterpret_cast<uintptr_t>(d_x) & 15) || (reinterpret_cast<uintptr_t>(d_y) & 15))
        return EP_ERR_BAD_ARG;
    if (reinterpret_cast<uintptr_t>(d_tables) & 255) return EP_ERR_SCRATCH;
    if (I.table_K[0] == 0 || I.table_min[0] < 0 || int64_t(I.table_min[0]) + I.table_K[0] > 2) return EP_ERR_BAD_STREAM;
    // one tile per row (a warp decodes a row), whole groups per row, tables in shared memory
    if (I.b != 11 || !fits_smem_tables(I) || I.V != I.C / 8 || I.C % 256 || T > 32 ||
        I.total_words >= (1ull << 30) || uint64_t(I.R) * I.C >= (1ull << 32))
        return EP_ERR_UNSUPPORTED;
    const int sms = num_sms();
    if (sms <= 0) return EP_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    GemmParams P;
    std::memset(&P, 0, sizeof(P));
    JobParams &J = P.J;
    J.stream = static_cast<const uint8_t *>(d_stream);
    J.tile_index = static_cast<const uint32_t *>(d_tile_index);
    J.scales = d_row_scales;
    J.lut_image = static_cast<const uint32_t *>(d_tables);
    J.off_payload = I.off_payload;
    J.total_words = uint32_t(I.total_words);
    J.n_vec = uint32_t(uint64_t(I.R) * (I.C / 8));
    J.per_row = I.C / 8;
    J.V = I.V;
    J.n_tiles = I.n_tiles;
    J.tile_cnt = I.n_tiles;
    J.row_max = I.R - 1u;
    fill_table_params(J, I);
    P.y = d_y;
    P.T = T;
    P.Tpad = T <= 16 ? 16u : 32u;
    P.R = I.R;
    // rows spread evenly over the SMs, and a CTA's rows evenly over the fewest steps (a step lasts as long as its warps share an
    // SM's issue slots; 16 tokens, us, even steps / steps of 30 and a rest: 70 rows per SM of 10240 x 3840 53.5 / 58.4, 31 rows of 2048
    // columns 19.7 / 24.0, 50 23.0 / 24.5, 62 29.8 / 34.1)
    P.rows_per_cta = (I.R + uint32_t(sms) - 1u) / uint32_t(sms);
    const uint32_t most = ep::gemm_rows_per_step(T, P.rows_per_cta, I.C);
    P.steps = (P.rows_per_cta + most - 1u) / most;
    P.rows_per_step = (P.rows_per_cta + P.steps - 1u) / P.steps;
    P.groups = I.C / 256u;
    if (I.n_tiles != I.R) return EP_ERR_BAD_ARG;
    const auto kernel = P.Tpad == 16u ? (most == 30u ? ep_decode_gemm_kernel<16, 30> : ep_decode_gemm_kernel<16, 24>)
                                      : (most == 30u ? ep_decode_gemm_kernel<32, 30> : ep_decode_gemm_kernel<32, 24>);
    const uint32_t smem = P.Tpad == 16u ? (most == 30u ? GemmShape<16, 30>::kSmem : GemmShape<16, 24>::kSmem)
                                        : (most == 30u ? GemmShape<32, 30>::kSmem : GemmShape<32, 24>::kSmem);
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return EP_ERR_CUDA;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        if (cudaFuncSetAttribute(ep_decode_gemm_kernel<16, 30>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(GemmShape<16, 30>::kSmem)) != cudaSuccess ||
            cudaFuncSetAttribute(ep_decode_gemm_kernel<16, 24>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(GemmShape<16, 24>::kSmem)) != cudaSuccess ||
            cudaFuncSetAttribute(ep_decode_gemm_kernel<32, 30>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(GemmShape<32, 30>::kSmem)) != cudaSuccess ||
            cudaFuncSetAttribute(ep_decode_gemm_kernel<32, 24>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(GemmShape<32, 24>::kSmem)) != cudaSuccess)
            return EP_ERR_CUDA;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    const uint32_t grid = (I.R + P.rows_per_cta - 1u) / P.rows_per_cta;
    // x as a two-dimensional tensor for the copy engine: boxes of 64 columns (128 bytes, the swizzle span) x Tpad rows
    static EncodeTiledFn encode = nullptr;
    if (!encode) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
            qres != cudaDriverEntryPointSuccess)
            return EP_ERR_CUDA;
        encode = reinterpret_cast<EncodeTiledFn>(fn);
    }
    CUtensorMap x_map;
    const cuuint64_t dims[2] = {I.C, T}, strides[1] = {cuuint64_t(I.C) * 2u};
    const cuuint32_t box[2] = {64u, P.Tpad}, estr[2] = {1u, 1u};
    if (encode(&x_map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(d_x), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return EP_ERR_CUDA;
    const uint32_t threads = 32u * (2u + P.rows_per_step < kMinWarps ? kMinWarps : 2u + P.rows_per_step);
    return launch_next(kernel, grid, threads, smem, st, P, x_map) == cudaSuccess ? EP_OK : EP_ERR_CUDA;
}

extern "C" int ep_last_device_status(void *stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaStreamSynchronize(st) != cudaSuccess) return EP_ERR_CUDA;
    unsigned int v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_ep_status, sizeof(v)) != cudaSuccess) return EP_ERR_CUDA;
    if (v && cudaMemcpyToSymbol(g_ep_status, &zero, sizeof(zero)) != cudaSuccess) return EP_ERR_CUDA;
    return v ? EP_ERR_BAD_STREAM : EP_OK;
}

// ---- decode without a caller-provided scratch buffer ----------------------------------------------------
// For callers that cannot allocate device memory when they need to decode (they were given input and
// output buffers by a framework that owns the allocator, or an allocation would stall the device in the
// middle of serving).  The large-table path then builds its tables in this fixed area instead of in
// caller scratch.  One area per device, shared by every call: calls that overlap on the GPU race on it.
namespace {

constexpr size_t kStaticTableBytes = size_t(EP_NUM_TABLES) * (size_t(1) << EP_STATIC_MAX_B) * 4u;   // 557 056
static __device__ __align__(256) unsigned char g_ep_static_tables[kStaticTableBytes];

// In host code `g_ep_static_tables` is only a handle for the runtime, not an address a kernel could use:
// the device address is asked for once per device, with that device current.
void *g_static_tables_addr[64] = {};

int static_tables_address(void **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return EP_ERR_CUDA;
    if (dev < 0 || dev >= 64) return EP_ERR_UNSUPPORTED;
    if (!g_static_tables_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_ep_static_tables) != cudaSuccess || !p) return EP_ERR_CUDA;
        g_static_tables_addr[dev] = p;
    }
    *out = g_static_tables_addr[dev];
    return EP_OK;
}

}  // namespace

extern "C" int ep_decode_tensor_static(const ep_info *info, const void *d_stream, const void *d_tile_index,
                                       const float *d_row_scales, int32_t out_dtype, void *d_out, void *stream) {
    if (!info) return EP_ERR_BAD_ARG;
    void *tables = nullptr;
    size_t bytes = 0;
    if (ep_decode_scratch_bytes(info) != 0) {
        if (info->b > EP_STATIC_MAX_B) return EP_ERR_STATIC_LIMIT;   // tables of 2^b slots would not fit the built-in area
        const int rc = static_tables_address(&tables);
        if (rc) return rc;
        bytes = kStaticTableBytes;
    }
    return ep_decode_tensor(info, d_stream, d_tile_index, d_row_scales, out_dtype, d_out, tables, bytes, stream);
}

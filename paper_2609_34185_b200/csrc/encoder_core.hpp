// Shared pieces of the EntroPack encoder: the seventeen-table model, the stored-size estimate,
// the row sampler, blob assembly, and the search driver (Algorithm 1 plus the full-tensor rate
// correction) that runs on top of either back end - host threads (encoder.cpp) or CUDA kernels
// (encode_gpu.cu).  Both back ends produce byte-identical streams for the same input.
#pragma once
#include <cstdint>
#include <memory>
#include <new>
#include <utility>
#include <vector>

#include "stream.hpp"

// allocator whose resize() leaves new bytes uninitialised (a blob of tens of MB is written exactly once)
template <class T>
struct ep_no_init_allocator : std::allocator<T> {
    template <class U> struct rebind { using other = ep_no_init_allocator<U>; };
    ep_no_init_allocator() = default;
    template <class U> ep_no_init_allocator(const ep_no_init_allocator<U> &) {}
    template <class U> void construct(U *p) { ::new (static_cast<void *>(p)) U; }
    template <class U, class... A> void construct(U *p, A &&...a) { ::new (static_cast<void *>(p)) U(std::forward<A>(a)...); }
};

// Host storage of a stored representation.  By default ordinary heap memory; a back end may install its
// own source (the GPU back end: page-locked memory, which the device copies into at full bus speed and
// which a later upload reads at full speed too) before the blob is assembled.
struct ep_blob {
    std::vector<uint8_t, ep_no_init_allocator<uint8_t>> heap;
    uint8_t *ext = nullptr;                                  // storage obtained through `acquire`
    size_t ext_size = 0, ext_cap = 0;
    uint8_t *(*acquire)(size_t n, size_t *cap) = nullptr;    // nullptr on failure
    void (*release)(uint8_t *p, size_t cap) = nullptr;
    ep_encode_report report{};

    ep_blob() = default;
    ep_blob(const ep_blob &) = delete;
    ep_blob &operator=(const ep_blob &) = delete;
    ~ep_blob() { if (ext && release) release(ext, ext_cap); }
    // n bytes of uninitialised storage (replaces what the blob held); nullptr if the source has none
    uint8_t *allocate(size_t n) {
        if (acquire) {
            if (ext && release) release(ext, ext_cap);
            ext_size = ext_cap = 0;
            ext = acquire(n, &ext_cap);
            if (!ext) return nullptr;
            ext_size = n;
            return ext;
        }
        heap.resize(n);
        return heap.data();
    }
    // the blob has only n of the bytes that were allocated
    void shrink(size_t n) { if (ext) ext_size = n; else heap.resize(n); }
    const uint8_t *data() const { return ext ? ext : heap.data(); }
    uint8_t *data() { return ext ? ext : heap.data(); }
    size_t size() const { return ext ? ext_size : heap.size(); }
};

#ifdef __CUDACC__
#define EP_HOST_DEVICE __host__ __device__
#else
#define EP_HOST_DEVICE
#endif

namespace ep {

constexpr double kEta = 1e-12;

int resolve_threads(int requested);

// ---- Sec. 3.3: the seventeen categorical tables -------------------------------------------------
struct Table {
    int32_t lo = 0;
    std::vector<uint64_t> n;   // counts over [lo, lo + K)
    std::vector<uint32_t> f;   // b-bit frequencies
    std::vector<uint32_t> F;   // exclusive prefix sums, K + 1 entries
    uint64_t total = 0;
    uint32_t K() const { return uint32_t(n.size()); }
    uint32_t observed() const;
};

struct Model {
    Table t[EP_NUM_TABLES];
    void count(const int32_t *fields, uint64_t nvec, int threads);          // from (c, z1..z7, m) tuples
    // from counts laid out table after table: K[t] counts of the values lo[t] .. lo[t] + K[t] - 1
    void from_counts(const int32_t *lo, const uint32_t *K, const uint32_t *counts);
    void normalise(int b);                                                   // integer frequencies summing to 2^b
    double cross_entropy_bits(int b) const;                                  // Eq. 8
    uint64_t section_bytes() const;
    uint32_t worst_observed() const;                                         // largest alphabet over all tables
    uint32_t worst_coordinate_observed() const;                              // A_max: over the 16 coordinate tables
};

// Eq. 10-11: estimated stored bits of nvec vectors in `rows` rows under model m
double estimate_bits(const Model &m, int b, uint64_t nvec, uint64_t rows, uint32_t V, double retained, double *cce_out);

// The CUDA back end's tile coder looks a symbol up by (coset, field, value): per field the tables of both cosets cover the same
// values, from the lower to the higher end of the two, so that coset 1's entries follow coset 0's at one distance; the
// coset's own two entries come last.  The ranges of the two cosets need not meet - a few large blocks in a tensor of
// zeros: one coset at -3873, the other at 3872 - so what bounds the entries is not the number of symbols but the
// values a field can have.
constexpr int kHistBins = 8192;          // values per table that the CUDA back end counts
constexpr uint32_t kCoderEntries = 2u * 8u * kHistBins + 2u;
struct CoderLayout {
    int32_t lo[9] = {};                  // field k's lowest value (k = 1 .. 8) and
    uint32_t first[9] = {};              // where its entry is
    uint32_t size = 0;                   // entries per coset
    uint32_t entries() const { return 2u * size + 2u; }
};
inline CoderLayout coder_layout(const Model &m) {
    CoderLayout L;
    for (int k = 1; k < 9; ++k) {
        int32_t hi = 0;
        bool any = false;
        for (int c = 0; c < 2; ++c) {
            const Table &tb = m.t[table_id(c, k)];
            if (!tb.K()) continue;
            const int32_t end = tb.lo + int32_t(tb.K());
            L.lo[k] = any && L.lo[k] < tb.lo ? L.lo[k] : tb.lo;
            hi = any && hi > end ? hi : end;
            any = true;
        }
        L.first[k] = L.size;
        L.size += uint32_t(hi - L.lo[k]);
    }
    return L;
}

// Rate correction in a back end of its own arithmetic: how far, relatively, the next scale 2^(log_s + off_target / per_doubling)
// can be from run_encode's if log2 and exp2 are within one unit in the last place there and here (two between them;
// u = 2^-52), and everything else is rounded as there.  The secant divides by log_s - last_log_s, which scales next
// to each other make as small as 2^-23.5: then two such units of log_s are 1e-8 of the slope.
EP_HOST_DEVICE inline double next_scale_error(double log_s, double last_log_s, bool secant, double off_target, double per_doubling) {
    const double u = 2.220446049250313e-16;
    const double size = log_s < 0 ? -log_s : log_s, last = last_log_s < 0 ? -last_log_s : last_log_s;
    double slope = 2.0 * u;                          // relative, clamping to [1/2, 4] does not add to it
    if (secant) {
        const double moved = log_s < last_log_s ? last_log_s - log_s : log_s - last_log_s;
        const double off = 2.0 * u * (size + last) + u * moved;
        if (!(off < 0.25 * moved)) return 1.0;       // says nothing
        slope += 1.34 * off / moved;                 // 1 / (1 - 1/4)
    }
    double step = off_target / per_doubling;
    if (step < 0) step = -step;
    const double exponent = 2.0 * u * size + step * (slope + 2.0 * u) + u * (size + step);
    return 0.7 * exponent + 8.0 * u;                 // ln 2, exp2 on either side and the roundings of a comparison
}

// A pass of the CUDA back end's search counts `scales` scales, each with the same number of the grid's CTAs.  The CTAs that are left over do
// nothing, and nobody waits for them: one that starts late - another stream's kernel, or another encode, held its SM - may read the
// number of scales after the pass's last CTA has stored the next pass's.  So the number is stored together with its pass, and a CTA takes a
// number of any other pass for none.  (The others' numbers and scales stand until they have all arrived.)  One CTA per SM, but never fewer than
// a pass may have scales: a process limited to a share of the GPU may see fewer SMs than that.
constexpr uint32_t kMostScales = 15;
inline uint32_t pass_grid(uint32_t sms) { return sms > kMostScales ? sms : kMostScales; }
struct PassShare { uint32_t scale, part, ctas; };        // this CTA's scale (>= scales: left over), its share of the blocks, of how many
EP_HOST_DEVICE inline PassShare pass_share(uint32_t grid, uint32_t cta, uint32_t scales, uint32_t n_blocks) {
    const uint32_t fit = grid / scales, useful = (n_blocks + 255u) / 256u, ctas = fit < useful ? fit : useful;
    return {cta / ctas, cta % ctas, ctas};
}
EP_HOST_DEVICE inline uint32_t scales_word(uint32_t pass, uint32_t scales) { return pass * 16u + scales; }
EP_HOST_DEVICE inline uint32_t scales_of(uint32_t word, uint32_t pass) {
    const uint32_t scales = word - pass * 16u;
    return scales <= kMostScales ? scales : 0u;
}

// App. "Scale-search settings": complete rows, shape-dependent seed, sorted
std::vector<uint32_t> sample_rows(uint32_t R, uint32_t C, uint32_t budget_vectors);

// Where the sections of a stored representation lie.  Scales, tile index and payload are back to back.
struct BlobLayout { uint64_t off_tables, off_scales, off_tiles, off_payload, total; };

// Allocates a blob for total_words payload words and writes its header and tables; the three sections after
// off_scales are left to the caller.  If it turns out to have fewer words, end_blob corrects the size.
int begin_blob(const Model &m, uint32_t R, uint32_t C, int b, uint32_t V, float s_info, uint64_t total_words, ep_blob *out,
               BlobLayout *at);
void end_blob(const BlobLayout &at, uint64_t total_words, ep_blob *out);

// How many payload words to lay a blob out for before the tile coder is done, given C_CE of the final tables, the words' area
// and the bytes before the payload: a few more than the entropy says (coding loses about 1e-5 of it, and a tile's states
// keep some bits), never more than the area holds or a blob can have (its section offsets and its size are 32-bit).
// 0: the tiles have more than a blob can hold whatever their states keep (at most 16 bits each).
inline uint64_t payload_room(double cce_bits, uint64_t n_tiles, uint64_t area_words, uint64_t bytes_before) {
    const uint64_t bytes = (1ull << 32) - 1u, most = bytes_before < bytes ? (bytes - bytes_before) / 2u : 0u;
    if (0.98 * cce_bits / 16.0 - double(kStates * n_tiles) > double(most)) return 0;
    const uint64_t guess = uint64_t(cce_bits / 16.0 * 1.001) + 8u * n_tiles + 256u, room = guess < area_words ? guess : area_words;
    return room < most ? room : most;
}

// header + tables + scales + tile index + payload; `states` holds 32 words per tile, tile t's payload is
// tile_words[t] .. + tile_len[t].
int assemble_blob(const Model &m, uint32_t R, uint32_t C, int b, uint32_t V, const float *sigma, float s_info,
                  const uint32_t *states, const uint16_t *const *tile_words, const uint32_t *tile_len, ep_blob *out);

// One bisection of Algorithm 1 for a back end that runs it whole.
struct SearchJob {
    double target_bpp;
    int b;
    uint32_t V;
    uint64_t sample_vectors;     // vectors in the row sample
    size_t sample_rows;
};
struct SearchResult {
    float s = 0.0f;              // the scale the bisection, or the rate correction after it, ends on
    bool polished = false;       // the rate correction is done as well
    Model last;                  // counts of the last candidate whose rate was evaluated
    bool has_last = false;
    Model full;                  // counts of the whole tensor at s (quantisation kept, as by count_full)
};

// What a back end must provide.  Each call returns an ep_status.
struct EncodeBackend {
    virtual ~EncodeBackend() {}
    virtual int prepare(const std::vector<uint32_t> &sample) = 0;   // row RMS; remember the row sample
    virtual int count_sample(float s, Model &m) = 0;                // quantise the sample at s, count its fields
    virtual int count_full(float s, Model &m) = 0;                  // quantise the whole tensor at s (kept), count
    // the bisection of Algorithm 1 on the row sample, the full-tensor pass at the scale it ends on and, if that fits the
    // tables, the rate correction, in one go.
    // *done = false: not supported, or a decision the back end will not take; the driver then runs it step by step
    virtual int search(const SearchJob & /*job*/, const ep_encode_opts & /*o*/, SearchResult & /*r*/, bool *done) { *done = false; return EP_OK; }
    // refit the row scales of the kept quantisation (Eq. 13), encode the tiles under the normalised full-tensor model m
    // and assemble the blob; the driver has work of its own between the two calls
    virtual int begin_finish(float s, int b, uint32_t V, const Model &m) = 0;
    virtual int end_finish(float s, int b, uint32_t V, const Model &m, double cce_bits, ep_blob *out) = 0;
    // per-row rate-distortion refinement of the kept quantisation (Sec. 3.5, Alg. 2); on success `m` holds the
    // counts of the refined fields and end_finish() uses the refined row scales.  Optional.
    virtual int refine(float /*s*/, int /*b*/, uint32_t /*V*/, const ep_encode_opts & /*o*/, Model & /*m*/) { return EP_ERR_UNSUPPORTED; }
};

// the K nested candidate ratios of Alg. 2: 1 first, then log-midpoints of the widest remaining interval of [0.70, 1.45]
std::vector<double> rdo_ratios(int K);

// Algorithm 1, the rate-correction stage and the final packing over a back end.
int run_encode(EncodeBackend &be, uint32_t R, uint32_t C, double target_bpp, const ep_encode_opts &o, ep_blob **out);

}  // namespace ep

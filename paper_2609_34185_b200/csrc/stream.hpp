// Stored-representation layout helpers shared by the host encoder, the validator and the
// decode launcher of the library.  Byte layout: see include/entropack.h.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#include "entropack.h"

namespace ep {

constexpr uint32_t kMagic = 0x314B5045u;  // "EPK1"
constexpr uint32_t kHeaderBytes = 64;
constexpr uint32_t kStates = 32;          // J
constexpr uint32_t kTileRecordBytes = 4 * kStates + 4;
constexpr uint32_t kStateLow = 1u << 15;  // states live in [2^15, 2^31)
constexpr uint32_t kDecodeTilesPerCta = 32;  // tiles one CTA of the decode kernel works on at a time (one per warp)

template <class T>
inline T load_le(const uint8_t *p) {
    T v;
    std::memcpy(&v, p, sizeof(T));  // little-endian hosts only (x86-64, aarch64)
    return v;
}
template <class T>
inline void store_le(uint8_t *p, T v) {
    std::memcpy(p, &v, sizeof(T));
}

// table id of field k (0 = coset, 1..7 = z_k, 8 = m) under coset c
inline int table_id(int c, int k) { return k == 0 ? 0 : 1 + 8 * c + (k - 1); }

inline uint64_t table_section_bytes(const uint32_t K[EP_NUM_TABLES]) {
    uint64_t k = 0;
    for (int t = 0; t < EP_NUM_TABLES; ++t) k += K[t];
    return (8ull * EP_NUM_TABLES + 2ull * k + 3ull) & ~3ull;
}

// Few tiles per SM: does the decode loop that guesses (EP_BODY11_GUESS) pay, for a stream of `bits` payload bits per symbol and
// `symbols` symbols per coordinate table on average, `tiles` tiles of `blocks` blocks per SM?
// The guess saves 14 % of a group's time with up to 4 tiles and 8 with up to 8 (beyond, its ten extra instructions per step cost more
// than they save); a group whose guess fails is decoded twice, and a launch lasts as long as its unluckiest tile.  So the shorter the
// tiles, the fewer failures they bear, and the failures grow with the rate and with the share of rare symbols: Laplace rows
// repeat as many groups at 3.6 bits as Gaussian ones at 4.4, one in 17.  To BF16, graph of launches, us, with / without:
//   Gaussian      256 blocks: 4 tiles 2.4 bits 7.2 / 7.5, 3.6 7.9 / 7.6; 8 tiles 2.0 bits 7.6 / 7.7, 3.2 8.1 / 7.8
//                 512: 4 tiles 3.4 bits 11.8 / 12.4, 4.0 12.4 / 12.4; 8 tiles 2.8 bits 12.7 / 12.9, 3.6 13.3 / 12.8
//                 1024: 4 tiles 4.0 bits 20.8 / 22.0, 4.2 22.8 / 22.0; 8 tiles 3.4 bits 22.2 / 23.0, 4.0 23.4 / 23.0
//                 1792: 4 tiles 4.2 bits 34.5 / 36.3, 4.6 36.9 / 36.3; 8 tiles 3.8 bits 36.4 / 38.0, 4.2 38.4 / 38.0
//                 3640: 4 tiles 4.2 bits 68.2 / 73.3, 4.6 71.9 / 73.3; 8 tiles 4.2 bits 77.7 / 78.5, 4.4 79.9 / 78.6
//   Laplace       512: 4 tiles 2.4 bits 12.3 / 12.4, 3.2 13.0 / 12.4; 8 tiles 2.0 bits 12.6 / 12.9, 2.8 13.4 / 12.9
//                 1024: 4 tiles 3.2 bits 20.9 / 21.9, 3.7 22.6 / 21.9; 8 tiles 2.8 bits 22.7 / 22.8, 3.5 24.5 / 22.9
//                 1792: 4 tiles 3.5 bits 35.0 / 36.2, 4.1 39.4 / 36.2; 8 tiles 3.2 bits 37.5 / 37.9, 4.1 42.8 / 38.1
//                 3640: 4 tiles 3.9 bits 72.7 / 73.3, 4.5 82.9 / 73.3; 8 tiles 3.5 bits 77.3 / 78.6, 3.9 81.7 / 78.5
// Gaussian rows with outliers bear what Gaussian ones do, but have alphabets as wide as heavy-tailed ones: log2 of the mean
// alphabet is 1.2 - 1.7 above the rate for Gaussian rows, 2.0 - 2.8 for Laplace, 2.2 - 3.8 for Student-t, 2.2 - 2.4 with outliers
// (128 thousand to 34 million weights).  So the line for wide alphabets lies between what those three bear.  Over twelve sizes of tile, 1.6 to
// 4.6 bits, eleven tile counts and four output types the lines are, on average, 0.1 % (Gaussian), 0.3 % (outliers) and 0.2 - 1.3 % (Laplace,
// Student-t: eight and four tiles) behind the better of the two; one line for all rows, 4.2 bits (4.5 above 1024 blocks) and, from
// 512 blocks on, 4.1 bits, was 0.4 - 0.9, 0.6 - 1.2 and 2.4 - 4.4 %.
inline bool guess_pays(uint32_t tiles, uint32_t blocks, double bits, double symbols) {
    if (tiles > 8u) return false;
    const double root = std::sqrt(double(blocks));
    const bool wide = std::log2(symbols) > bits + 1.85;
    if (tiles <= 4u) return bits <= 5.1 - 29.0 / root && !(wide && bits > 4.2);
    return bits <= 4.9 - (wide ? 48.0 : 34.0) / root && !(wide && bits > 3.6);
}

// ep_decode_gemm: most rows of W per step, 30 or 24 (what each leaves room for: GemmShape), for CTAs of `rows` rows.
// The one that takes fewer steps.  4096 columns at 4 bpp, 32 tokens, us, 24 / 30: 10 rows per SM 19.9 / 20.3, 23: 23.5 / 24.0, 28:
// 37.0 / 26.2, 56: 57.5 / 48.5, 70: 65.6 / 63.9, 91: 79.5 / 81.0, 120: 108.2 / 91.9.
// With equal steps 24 for 17 to 32 tokens (four units of x), and up to 16 tokens for the larger payload rings, but for short rows, for which
// they ask for more than a row has.  16 tokens, 4 bpp, graph of launches, us, 24 / 30: 256 columns 16 rows 4.9 / 4.7, 512 columns
// 20 rows 5.9 / 5.7 (one token 6.0 / 5.8), 768 columns 70 rows 14.7 / 15.4 (one token 20 rows 7.0 / 6.8), 1024 columns 70 rows 17.4 / 17.9.
inline uint32_t gemm_rows_per_step(uint32_t tokens, uint32_t rows, uint32_t columns) {
    const auto steps = [rows](uint32_t most) { return (rows + most - 1u) / most; };
    return steps(30u) < steps(24u) || (tokens <= 16u && columns <= 512u) ? 30u : 24u;
}

int parse_info(const void *blob, size_t n, ep_info *out);

}  // namespace ep

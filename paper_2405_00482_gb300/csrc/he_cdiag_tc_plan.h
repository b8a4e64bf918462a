// he_cdiag_tc_plan.h -- sizes of the tensor-core ciphertext-diagonal product (he_cdiag_tc.cu): tiles,
// passes over the diagonals, slices of tiles and the scratch that holds a slice's operands.  Plain C++,
// without CUDA, so that a host test can walk every pass.
#pragma once
#include <stdint.h>

#include <algorithm>

constexpr int TC_COLS = 128;                // weight columns per tile (the instruction's M)
constexpr int TC_ROWS = 64;                 // rows of a tile: 2 components x 32 coefficients
constexpr int TC_KC = 64;                   // indices s per chunk (128 bytes of bfloat16: one swizzle row)
constexpr int TC_DIAGS = 256;               // diagonals per pass: 255^2 256 < 2^24
constexpr int TC_A_BYTES = TC_COLS * TC_KC * 2, TC_B_BYTES = TC_ROWS * TC_KC * 2;
constexpr int64_t TC_SLICE_BYTES = 96ll << 20;  // of the 126 MB L2
constexpr int TC_MAX_MOD = 15;
// odd, pairwise coprime, below 512
constexpr int TC_MODULI[TC_MAX_MOD] = {511, 509, 507, 503, 499, 493, 491, 487, 485, 479, 473, 467, 463, 461, 457};

// moduli count for the prime q: prod p_i > 2.01 TC_DIAGS q (q / 2); 0 where the three 20-bit digits
// of the reconstruction do not hold a residue
inline int tc_moduli(uint64_t q) {
    if (q >> 60) return 0;
    long double need = 2.01L * TC_DIAGS * (long double)q * ((long double)q / 2), have = 1;
    for (int m = 0; m < TC_MAX_MOD; ++m) {
        have *= TC_MODULI[m];
        if (have > need) return m + 1;
    }
    return 0;
}

// Diagonals from which the tensor cores take a product of n weight rows by K columns (8 and more) sooner
// than the integer form.  The integer form's time is proportional to the diagonals and the blocks of 128
// columns; that of the tensor cores, up to a window of 64 diagonals, to the moduli (three-digit limbs
// cost 1.6 of the others in conversion and reconstruction), to the window's chunks (one for n <= 32,
// more as a window of n = 64 and more begins anywhere in a chunk) and, for the longest periods, to the
// weights, which outgrow L2.  More columns fill the same instructions; columns that are no multiple of 8
// slow the integer form's loads.  The factors are fitted to both forms' times over N = 2^12 (2 limbs), 2^13
// (3) and 2^14 (3 and 7), 8 to 200 columns, 8 to 8192 rows and 4 to 32 diagonals: the chosen form takes
// 1.004 times the faster one's time on average, 1.16 at worst.  At N = 2^14, 7 limbs, in us, tensor cores /
// integer form for 8, 12, 16, 20 and 24 diagonals, then the line:
//     8 columns, n =   16: 437/305 437/401 440/503                    14
//     8 columns, n =  256: 509/296 517/391 522/493 526/593 527/690    18
//     8 columns, n = 8192: 542/296 552/392 567/495 585/593 611/691    20
//    30 columns, n =  256: 591/429 600/544 605/664 608/780            15
//   128 columns, n =  256: 863/749 871/855 876/969 881/1077 883/1184  15
inline int tc_min_diags(const uint64_t *primes, int nl, int64_t n, int64_t K) {
    int64_t cost = 0;  // in fifths of a two-digit limb's modulus
    for (int u = 0; u < nl; ++u) cost += tc_moduli(primes[u]) * (primes[u] >> 40 ? 8 : 5);
    const int rows = n <= 32 ? 7 : n <= 64 ? 8 : n <= 2048 ? 9 : 10;  // sixths of a diagonal per modulus
    const int cols = (K < 96 ? 5 : K <= 128 ? 4 : 3) * (K % 8 ? 4 : 5);  // twenty-fifths
    const int64_t den = 5 * 6 * 25 * (int64_t)nl;
    return (int)((cost * rows * cols + den - 1) / den);
}

// chunks of the longest window of cnt diagonals: its start is rounded down to a whole chunk from the
// tile's first block, a multiple of the span (at most 32) of its blocks: 64 - span, span - 1 and the
// diagonals
inline int tc_chunks(int cnt) { return (TC_KC - 1 + cnt + TC_KC - 1) / TC_KC; }

// the pass over the diagonals i0 .. i0 + cnt of n_ct, on operands of up to `mods` moduli
struct TcPass {
    int cnt, chunks;
    int64_t tile_bytes;  // operand blocks of a tile: [modulus][chunk][64 rows x 128 bytes]
    int slice;           // tiles of a slice: a whole number per SM, their operands at most TC_SLICE_BYTES
                         // (one tile per SM at least), so that they are still in L2 when the product kernel
                         // reads them
};
inline TcPass tc_pass(int sms, int mods, int n_ct, int i0) {
    TcPass p;
    p.cnt = std::min(TC_DIAGS, n_ct - i0);
    p.chunks = tc_chunks(p.cnt);
    p.tile_bytes = (int64_t)mods * p.chunks * TC_B_BYTES;
    p.slice = sms * (int)std::max<int64_t>(1, TC_SLICE_BYTES / (p.tile_bytes * sms));
    return p;
}

// A term y h of a digit's sum (h a signed digit, |h| <= 2^19; |y| <= 256), y as the bits of the float
// 1.5 2^23 + y: TC_MAGIC_BITS + y.  The products and sums wrap mod 2^32; started at tc_digit_init, less
// the bias of every term to come, a sum of at most TC_MAX_MOD terms ends as the exact value below 2^31.
constexpr uint32_t TC_MAGIC_BITS = 0x4B400000u;
#ifdef __CUDACC__
__host__ __device__
#endif
inline uint32_t tc_digit_add(uint32_t sum, uint32_t y_bits, int32_t h) { return sum + y_bits * (uint32_t)h; }
inline uint32_t tc_digit_init(uint32_t init, int32_t h) { return init - TC_MAGIC_BITS * (uint32_t)h; }

// operand scratch of a product of n_ct diagonals over `tiles` tiles: the largest slice of any pass.  A
// short last pass has smaller tiles but more of them in a slice, and can need more than a full one (10
// moduli, 152 SMs: 62 MB for 256 diagonals, 100 MB for the 44 left of 300).
inline int64_t tc_scratch_bytes(int sms, int tiles, int mods, int n_ct) {
    int64_t bytes = 0;
    for (int i0 = 0; i0 < n_ct; i0 += TC_DIAGS) {
        const TcPass p = tc_pass(sms, mods, n_ct, i0);
        bytes = std::max(bytes, std::min(p.slice, tiles) * p.tile_bytes);
    }
    return bytes;
}

// Which packed linears keep their expanded weights in shared memory (gemm_direct.cu).  Plain C++: sizes in, tile width out.
#pragma once
#include <cstdint>

namespace vitint {

constexpr uint32_t GD_RESIDENT_BYTES = 218u * 1024u;          // rings and resident weights of packed operands

// Both operands bit-packed alike (`bits` a code): what a K block of 128 codes costs is shared-memory traffic, three passes (packed
// in, packed out, expanded in) over each expanded operand and the tensor core's reads of both.  A CTA whose tiles lie in one
// column of tiles can expand their weights once and keep them: per K block 384 + columns cycles instead of 3 (128 + columns).
// Returns the tile width, a multiple of `block` columns, where that is the cheaper way than tiles of bn0 columns (0: nowhere): the
// weights fit beside two operand slots and two packed ones, and the grid, a whole number of CTAs for each column of tiles, wastes
// less than is won.  12,608 x 768 -> 3072 requantized (with the quantizer in front) 58.9 -> 49.3 us, 25,216 x 768 -> 2304
// 90.9 -> 78.4, 6304 x 768 -> 2000 34.5 -> 23.3 (with the ragged width); one tile a CTA gains nothing.
// The int32 bound on accumulators lets unsigned 2-bit codes have K up to 2^27, so sizes are formed in 64 bits.
inline int resident_tile_columns(int sms, int m_tiles, int k_blocks, int n, int bits, int block, int bn0, bool fp32_out) {
    const long long tiles0 = (long long)m_tiles * ((n + bn0 - 1) / bn0);
    if (tiles0 <= sms) return 0;
    // fp32 results are half bound by HBM: 12,608 x 384 -> 384 (0.76 of the cycles) gains, 25,216 x 768 -> 768 (0.83) is level
    long long best_t = (tiles0 + sms - 1) / sms * 3 * (128 + bn0) * (fp32_out ? 80 : 95) / 100;
    int best = 0;
    for (int bn = 256; bn >= block; bn -= block) {
        const int n_tiles = (n + bn - 1) / bn;
        const long long slots = 2ll * 128 * 128 + 2ll * (128 + bn) * 16 * bits, kept = (long long)k_blocks * bn * 128;
        if (n_tiles > sms || slots + kept > (long long)GD_RESIDENT_BYTES) continue;
        const long long per_column = sms / n_tiles, rounds = (m_tiles + per_column - 1) / per_column, t = rounds * (384 + bn) + 2 * bn;
        if (t < best_t) { best_t = t; best = bn; }
    }
    return best;
}

}  // namespace vitint

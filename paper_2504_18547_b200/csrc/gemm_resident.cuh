// Which packed linears keep their expanded weights in shared memory (gemm_direct.cu).  Plain C++: sizes in, tile width out.
#pragma once
#include <cstdint>

namespace vitint {

constexpr uint32_t GD_RING_BYTES = 200u * 1024u;
constexpr uint32_t GD_RESIDENT_BYTES = 218u * 1024u;          // rings and resident weights of packed operands

// Slots of the ring of packed tiles beside three operand slots, or two where three leave no room for two packed ones.
inline long long packed_slots(long long ring, long long operand_slot, long long packed_slot) {
    const int ns = 3 * operand_slot + 2 * packed_slot > ring ? 2 : 3;
    return (ring - ns * operand_slot) / packed_slot;
}

enum PackedEpilogue { PE_REQUANT, PE_GELU, PE_FP32 };

// Both operands bit-packed alike (`bits` a code): what a K block of 128 codes costs is shared-memory traffic, three passes (packed
// in, packed out, expanded in) over each expanded operand and the tensor core's reads of both.  A CTA whose tiles lie in one
// column of tiles can expand their weights once and keep them: per K block 384 + columns cycles instead of 3 (128 + columns).
// Returns the tile width, a multiple of `block` columns, where that is the faster way than tiles of bn0 columns (0: nowhere): the
// weights fit beside two operand slots and two packed ones, and the grid, a whole number of CTAs for each column of tiles, wastes
// less than is won.  12,608 x 768 -> 3072 requantized (with the quantizer in front) 58.9 -> 49.3 us, 25,216 x 768 -> 2304
// 90.9 -> 78.4, 6304 x 768 -> 2000 34.5 -> 23.3 (with the ragged width); one tile a CTA gains nothing.
//
// More rounds of tiles also cost more epilogues.  Both forms of 434 linears (2 and 4 bits, M 3000 .. 50,432, K 128 .. 1536, N 192 ..
// 4096) are told apart by rounds x (K blocks x (1.2 or 3 cycles x the above) + columns x E), E = 14 (requantize, 4 bits), 37 (2 bits),
// 55 (GELU): the 288 that are taken gain 6.5 % in the mean and lose 1.4 % at worst, the others would lose 2.7 % in the mean.  By
// shared-memory traffic alone 50,432 x 1024 -> 1024 went 77.0 -> 79.5 us, 25,216 x 640 -> 640 of 2 bits 18.4 -> 21.2, 25,216 x 192 ->
// 768 with GELU 21.6 -> 25.1.  fp32 results are half bound by HBM and need the packed ring's depth: taken with no more columns a
// CTA in all and no shallower a ring than three slots or the other form's (12,608 x 512 -> 2048 35.6 -> 28.5; without that
// 25,216 x 768 -> 2304 of 2 bits 61 -> 75, 12,608 x 768 -> 3072 49.9 -> 58.2).
// The int32 bound on accumulators lets unsigned 2-bit codes have K up to 2^27, so sizes are formed in 64 bits.
inline int resident_tile_columns(int sms, int m_tiles, int k_blocks, int n, int bits, int block, int bn0, PackedEpilogue epi) {
    const long long tiles0 = (long long)m_tiles * ((n + bn0 - 1) / bn0), rounds0 = (tiles0 + sms - 1) / sms, kb = k_blocks;
    if (tiles0 <= sms) return 0;
    auto kept = [&](int bn) { return kb * bn * 128; };
    auto rounds = [&](int bn) { const long long per_column = sms / ((n + bn - 1) / bn); return (m_tiles + per_column - 1) / per_column; };
    long long best_t = rounds0 * 3 * (128 + bn0) * (epi == PE_FP32 ? 80 : 95) / 100;
    int best = 0;
    for (int bn = 256; bn >= block; bn -= block) {
        const long long slots = 2ll * 128 * 128 + 2ll * (128 + bn) * 16 * bits;
        if ((n + bn - 1) / bn > sms || slots + kept(bn) > (long long)GD_RESIDENT_BYTES) continue;
        const long long t = rounds(bn) * (384 + bn) + 2 * bn;
        if (t < best_t) { best_t = t; best = bn; }
    }
    if (best == 0) return 0;
    if (epi == PE_FP32) {
        const long long deep = packed_slots(GD_RING_BYTES, 128 * 128 + bn0 * 128, (128 + bn0) * 16 * bits);
        return rounds(best) * best <= rounds0 * bn0 && packed_slots(GD_RESIDENT_BYTES - kept(best), 128 * 128, (128 + best) * 16 * bits) >= (deep < 3 ? deep : 3)
            ? best : 0;
    }
    const long long e = epi == PE_GELU ? 55 : bits == 2 ? 37 : 14;
    return 100 * rounds(best) * (12 * kb * (384 + best) + 10 * e * best) < 97 * rounds0 * (30 * kb * (128 + bn0) + 10 * e * bn0) ? best : 0;
}

}  // namespace vitint

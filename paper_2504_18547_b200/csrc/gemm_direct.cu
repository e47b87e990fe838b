// a2 + a3: the integer GEMM of gemm.cu with an epilogue laid out for the SM's shared-memory / L1 data pipe.
//
// With a thread per accumulator row (gemm.cu) every store of a warp walks 32 different rows and every parameter read serves
// two elements.  Here the epilogue reads the accumulators in the matrix-fragment layout (tcgen05.ld 16x256b: a thread holds
// a few columns of two rows), and the rows of the weight tile are PERMUTED by the TMA copy (a five-dimensional view of the
// weight matrix) so that the columns a thread holds are consecutive columns of the output:
//   codes  16 consecutive columns of a 64-column block: the per-column parameters are read once for four rows, and a
//          warp's 16-byte stores cover 64 contiguous bytes of 8 rows instead of 16 of 32;
//   norm   (QKV projection with the per-head quantizing LayerNorm) the Q and K tiles keep the weights' order, a thread walks a
//          row's 64 columns of a head;
//   fp32   8 consecutive columns of a 32-column block: a warp's 32-byte accesses of the residual and the result cover whole
//          128-byte lines, so nothing is staged through shared memory and the operand ring keeps the space.
// The arithmetic per element is that of gemm.cu, bit for bit.
//
// Measured against gemm_i8_kernel on the same operands (us, 4-bit codes, M = 25,216): 768 -> 2304 requantized 48.3 -> 40.1,
// 768 -> 3072 GELU 79.8 -> 72.1, 3072 -> 768 fp32 60.1 -> 55.5; at M = 197, where the tile width matters, 6.6 -> 4.5, 7.7 ->
// 4.9 and 15.0 -> 9.3, and 768 -> 768 fp32 9.9 -> 4.3.  What bounds it: the mainloop alone (no epilogue) takes 27.5, 35.9 and
// 36.2 us at M = 25,216, the epilogue alone 28, 63 (GELU: in the whole kernel the fp32 pipe is 53 % busy, the issue slots 57 %) and
// 38 us (its 155 MB); the two share the SM's issue slots and data pipe.
//
// The TMA and MMA warps run their loops as whole warps and elect a thread around each issue (see elect_one): 197 x 3072 -> 768 fp32
// 9.3 -> 6.6 us, 197 x 768 -> 768 4.4 -> 3.7, 197 x 768 -> 2304 4.6 -> 3.8, against one lane that runs the loop alone (a K block
// 0.27 us whatever the tile's width, now 0.17); 25,216 rows: 58.9 -> 57.0 (3072 -> 768), 40.6 -> 39.7, GELU 70.8 -> 68.1.
//
// Warps 0-15 epilogue (four per TMEM lane quarter, units of 16 rows x one column block in turn), 16 TMA, 17 MMA issue.  With
// bit-packed operands (PACKED) warps 8-15 expand them instead: two groups of four warps take K blocks in turn, and where both
// operands are packed alike the codes of a chunk keep the order in which masks and shifts produce them (the contraction does
// not mind), 12 operations for 32 codes instead of 20 and their sign left in the high bits.  12,608 x 768 -> 3072 of 4-bit
// packed codes, requantized: 81 -> 48 us (one group 63, two 58, reordered 48); 3072 -> 768 fp32 104 -> 52; 197 x 192 -> 576
// 7.6 -> 4.3.  Where a CTA keeps its columns' expanded weights (gemm_resident.cuh) only the activations are expanded tile by tile,
// 48 -> 39 us, and the eight epilogue warps beside them bound it: issue slots 42 % busy, load/store data pipe 34 % (53 and 56 % when
// both operands were expanded for every tile).  The byte-stored form takes 29 us.
#include "common.cuh"
#include "ptx.cuh"
#include "tile_ops.cuh"

#include "gemm_resident.cuh"

namespace vitint {
namespace {

// Epilogue warps of a group, unpack, TMA and MMA warps.  Eighteen warps leave a thread 96 registers; the norm kind takes groups
// of twelve epilogue warps, one for each lane quarter and head of a 192-column tile (two groups: 26 warps, 72 registers).
constexpr int GD_UNPACK_WARPS = 8;
__host__ __device__ constexpr int gd_epi_warps(int kind, bool packed) { return packed ? 16 - GD_UNPACK_WARPS : kind == EK_QKV_NORM ? 12 : 16; }
__host__ __device__ constexpr int gd_threads(int kind, bool packed, int groups = 1) {
    return (groups * gd_epi_warps(kind, packed) + (packed ? GD_UNPACK_WARPS : 0) + 2) * 32;
}

// Column block within which the weight rows are permuted: column 2q + 8g + e of the tensor-core block is output column
// (B/4) q + 2g + e, e < 2, q < 4, g < B/8.
__host__ __device__ constexpr int gd_block(int kind) { return kind == EK_DEQUANT ? 32 : 64; }

// Where column c of the tile keeps its parameters in shared memory: the four threads q of a row group read float4 number k
// of their columns at 64 consecutive bytes.
template <int BLK>
__device__ __forceinline__ int gd_param_slot(int c) {
    const int w = c & (BLK - 1), q = w / (BLK / 4), i = w & (BLK / 4 - 1);
    return (c - w) + (i >> 2) * 16 + q * 4 + (i & 3);
}

// What only some kernels need: the weights in their own order, for the norm kind's Q and K tiles and for a tile of codes that ends
// inside a column block (RAGGED).
struct NoExtra { int unused; };
struct OrderExtra { CUtensorMap map_w; };
template <int KIND, bool RAGGED> using DirectExtra = std::conditional_t<KIND == EK_QKV_NORM || RAGGED, OrderExtra, NoExtra>;

struct DirectBars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], acc_full[2], acc_empty[2], epi_sync[2], p_full[MAX_STAGES], p_empty[MAX_STAGES];
};

// One packed operand tile, `rows` rows of 16 C bytes -> rows of 128 int8 (128-byte swizzle), by 128 threads: thread t expands
// chunk t % C of rows t / C, t / C + 128 / C, ... (always the same row of an eight-row group, so nothing but two pointers
// changes along the way).
template <int C, int SGN, bool REORDER>
__device__ __forceinline__ void direct_unpack_tile(const uint8_t* src, uint8_t* dst, int rows, int t) {
    constexpr int STEP = 128 / C;
    const int r = t / C, sw = r & 7, oc = (t % C) * (8 / C);
    src += t * 16;
    dst += r * 128;
#pragma unroll 4
    for (; rows > 0; rows -= STEP, src += 2048, dst += STEP * 128)
        if (rows >= STEP || r < rows) {
            const uint4 in = *reinterpret_cast<const uint4*>(src);
            if (REORDER) expand_chunk_reordered<C, SGN>(in, dst, oc, sw);
            else expand_chunk<C, SGN>(in, dst, oc, sw);
        }
}
__device__ __forceinline__ void direct_unpack(int c, int is_signed, int reorder, const uint8_t* src, uint8_t* dst, int rows, int t) {
    if (c == 4) {
        if (reorder) is_signed ? direct_unpack_tile<4, 1, true>(src, dst, rows, t) : direct_unpack_tile<4, 0, true>(src, dst, rows, t);
        else is_signed ? direct_unpack_tile<4, 1, false>(src, dst, rows, t) : direct_unpack_tile<4, 0, false>(src, dst, rows, t);
    } else {
        if (reorder) is_signed ? direct_unpack_tile<2, 1, true>(src, dst, rows, t) : direct_unpack_tile<2, 0, true>(src, dst, rows, t);
        else is_signed ? direct_unpack_tile<2, 1, false>(src, dst, rows, t) : direct_unpack_tile<2, 0, false>(src, dst, rows, t);
    }
}

// Two accumulators (times 2^shift where signed codes were unpacked into the high bits of their bytes) -> float.  SMALL: the
// unscaled sums stay below 2^22, one integer addition each and a packed subtraction instead of the conversion instruction;
// otherwise 2^-shift rides on the multiplier.
template <bool SMALL, bool PACKED>
__device__ __forceinline__ f32x2 acc_to_float2(uint32_t v0, uint32_t v1, int shift) {
    if (SMALL && PACKED) { v0 = (uint32_t)((int)v0 >> shift); v1 = (uint32_t)((int)v1 >> shift); }
    if (SMALL) return f2_add(f2_pack(__uint_as_float(0x4B400000u + v0), __uint_as_float(0x4B400000u + v1)), f2_dup(-12582912.0f));
    return f2_pack((float)(int)v0, (float)(int)v1);
}

// The parameters of a thread's sixteen columns of a 64-column block.
template <bool GELU>
struct CodeParams {
    float4 a[4], b[4], q[GELU ? 4 : 1];
    __device__ __forceinline__ void load(const EpiParams& ep, int buf, int tile_col, int lane) {
        const int o = tile_col + (lane & 3) * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            a[k] = *reinterpret_cast<const float4*>(&ep.a[buf][o + 16 * k]);
            b[k] = *reinterpret_cast<const float4*>(&ep.b[buf][o + 16 * k]);
            if (GELU) q[k] = *reinterpret_cast<const float4*>(&ep.q[buf][o + 16 * k]);
        }
    }
};

// Four codes (bytes of a word, two's complement) of four consecutive columns of a row from their accumulators and parameters.
template <int KIND, bool SMALL, bool PACKED>
__device__ __forceinline__ uint32_t direct_quad(const GemmParams& P, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3, const float4& a,
                                                const float4& b, const float4& g4) {
    const f32x2 magic = f2_dup(12582912.0f), qp2 = f2_dup(P.out_qp);
    const float qn = P.out_qn, qp = P.out_qp;
    uint32_t c[4];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const f32x2 y = f2_fma(acc_to_float2<SMALL, PACKED>(p ? v2 : v0, p ? v3 : v1, P.shift), p ? f2_pack(a.z, a.w) : f2_pack(a.x, a.y),
                               p ? f2_pack(b.z, b.w) : f2_pack(b.x, b.y));
        float y0, y1, c0, c1;
        f2_unpack(y, y0, y1);
        if (KIND == EK_REQUANT_GELU) {
            // unsigned codes: the value arrives clamped to [0, 1] in units of Qp, and a negative y is code 0 whatever
            // its GELU: t = 0 there, the term is 1 and 2w - w = w < 0 saturates to 0
            float e0, e1, w0, w1, d0, d1;
            gelu_erfc_term2_pos(y0, y1, e0, e1);
            const f32x2 wq = f2_mul(y, p ? f2_pack(g4.z, g4.w) : f2_pack(g4.x, g4.y));
            f2_unpack(wq, w0, w1);
            f2_unpack(f2_add(wq, wq), d0, d1);
            const float u0 = __saturatef(fmaf(-w0, e0, d0)), u1 = __saturatef(fmaf(-w1, e1, d1));
            f2_unpack(f2_fma(f2_pack(u0, u1), qp2, magic), c0, c1);
        } else {
            f2_unpack(f2_add(f2_pack(fminf(fmaxf(y0, qn), qp), fminf(fmaxf(y1, qn), qp)), magic), c0, c1);
        }
        c[2 * p] = __float_as_uint(c0);                         // the code in two's complement is the low byte
        c[2 * p + 1] = __float_as_uint(c1);
    }
    return __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
}

// A tile that ends inside a column block: its weights lie in their own order (rows behind the last one zero) and a thread takes
// sixteen columns of its own row.  Parameters behind the last column are 0, and so are the codes, which fill the row's padding.
template <int KIND, bool SMALL, bool PACKED>
__device__ __forceinline__ void direct_codes_row(const GemmParams& P, uint32_t taddr, const EpiParams& ep, int buf, int tile_col,
                                                 long long row, bool row_ok, int col) {
    uint32_t v[16], w[4];
    ptx::tmem_ld16(taddr, v);
    ptx::tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 a = *reinterpret_cast<const float4*>(&ep.a[buf][tile_col + 4 * k]), b = *reinterpret_cast<const float4*>(&ep.b[buf][tile_col + 4 * k]);
        float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (KIND == EK_REQUANT_GELU) g4 = *reinterpret_cast<const float4*>(&ep.q[buf][tile_col + 4 * k]);
        w[k] = direct_quad<KIND, SMALL, PACKED>(P, v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3], a, b, g4);
    }
    if (!row_ok) return;
    uint8_t* const o = (uint8_t*)P.out + row * P.ld_out;
    store_row(o + ((col * P.out_c) >> 3), w, P.out_c);
    if (col + 16 >= P.N)
        for (long long off = (long long)(col + 16) * P.out_c >> 3; off + 4 <= P.ld_out; off += 4) *reinterpret_cast<uint32_t*>(o + off) = 0u;
}

// Requantizing epilogue of 16 rows x 64 columns, a thread's share two rows x 16 consecutive columns.
template <int KIND, bool SMALL, bool PACKED>
__device__ __forceinline__ void direct_codes(const GemmParams& P, const uint32_t (&v)[32], const CodeParams<KIND == EK_REQUANT_GELU>& cp,
                                             int lane, long long row0, int rows_valid, int n0) {
    const int r = lane >> 2, q = lane & 3;
    uint32_t w[2][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 g4 = KIND == EK_REQUANT_GELU ? cp.q[KIND == EK_REQUANT_GELU ? k : 0] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int h = 0; h < 2; ++h)                             // rows r and r + 8, columns 4k .. 4k + 3 of the thread's sixteen
            w[h][k] = direct_quad<KIND, SMALL, PACKED>(P, v[8 * k + 2 * h], v[8 * k + 2 * h + 1], v[8 * k + 4 + 2 * h], v[8 * k + 5 + 2 * h],
                                                       cp.a[k], cp.b[k], g4);
    }
    const int col = n0 + 16 * q;
    uint8_t* const o = (uint8_t*)P.out + (row0 + r) * P.ld_out + ((col * P.out_c) >> 3);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (r + 8 * h < rows_valid) {
            uint8_t* const oh = o + (h ? 8 * P.ld_out : 0);
            if (P.out_c == 8) {
                *reinterpret_cast<uint4*>(oh) = make_uint4(w[h][0], w[h][1], w[h][2], w[h][3]);
            } else if (P.out_c == 4) {
                uint32_t t[2];
                narrow4(w[h], t);
                *reinterpret_cast<uint2*>(oh) = make_uint2(t[0], t[1]);
            } else {
                *reinterpret_cast<uint32_t*>(oh) = narrow2(w[h]);
            }
            // row padding behind the last column of the matrix
            if (n0 + 64 >= P.N && q == 3)
                for (long long off = ((long long)P.N * P.out_c) >> 3; off + 4 <= P.ld_out; off += 4)
                    *reinterpret_cast<uint32_t*>((uint8_t*)P.out + (row0 + r + 8 * h) * P.ld_out + off) = 0u;
        }
    }
}

// Residual of 16 rows x 32 columns: rows r and r + 8, eight consecutive columns.
__device__ __forceinline__ void direct_residual(const GemmParams& P, int lane, long long row0, int rows_valid, int n0,
                                                float (&res)[2][8]) {
    const int r = lane >> 2, q = lane & 3;
    const float* const p = P.residual + (row0 + r) * P.ld_res + n0 + 8 * q;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (r + 8 * h < rows_valid) ptx::ld_global_32B(p + (h ? 8 * P.ld_res : 0), res[h]);
}

// fp32 epilogue of 16 rows x 32 columns.
template <bool SMALL, bool RES, bool PACKED>
__device__ __forceinline__ void direct_f32(const GemmParams& P, const uint32_t (&v)[16], const EpiParams& ep, int buf, int tile_col,
                                           int lane, long long row0, int rows_valid, int n0, const float (&res)[2][8]) {
    const int r = lane >> 2, q = lane & 3;
    float* const o = (float*)P.out + (row0 + r) * P.ld_out + n0 + 8 * q;
    float out[2][8];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float4 a = *reinterpret_cast<const float4*>(&ep.a[buf][tile_col + 16 * k + 4 * q]);
        const float4 b = *reinterpret_cast<const float4*>(&ep.b[buf][tile_col + 16 * k + 4 * q]);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int i = 8 * k + 4 * p + 2 * h, j = 4 * k + 2 * p;
                f32x2 y = f2_fma(acc_to_float2<SMALL, PACKED>(v[i], v[i + 1], P.shift), p ? f2_pack(a.z, a.w) : f2_pack(a.x, a.y),
                                 p ? f2_pack(b.z, b.w) : f2_pack(b.x, b.y));
                if (RES) y = f2_add(y, f2_pack(res[h][j], res[h][j + 1]));
                f2_unpack(y, out[h][j], out[h][j + 1]);
            }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (r + 8 * h < rows_valid) ptx::st_global_32B(o + (h ? 8 * P.ld_out : 0), out[h]);
}

// ---- QKV projection with the per-head quantizing LayerNorm of Section IV-C (Eq. 5 statistics, comparator of Fig. 5(b)) -----
// A thread owns the 64 channels of a head of one accumulator row.  It walks them in order through the recurrence of Eq. 5
//     delta = y_i - mu;  mu += delta / i;  S += delta * (y_i - mu)          (one rounded fp32 operation each)
// with y_i = fma(float(acc_i), s_x s_w[i], b_i), forms V = S + n*eps, reads the accumulators a second time and finds each level
// as Qn + number of references r with copysign(d*d, d) > V*r, d = y - mu (negated where the gain is negative): the count is
// guessed from d / sqrt(V) (folded from a uniform quantizer, the references are the signed squares of equally spaced points)
// and proven by two comparisons, formed exactly as defined, around it; where they fail all references are compared.  The fp32 Q
// and K never exist in memory.  Both passes are rolled loops over 16 columns: unrolled over the 64 their code streams through
// the instruction cache once per head, and that, not arithmetic, set the pace (one 197-row tile 9.8 us, of which the levels 6).
// 12,672 x 384 -> 1152 (DeiT-S width, batch 64, 3-bit): 49 -> 31 us, 197 x 192 -> 576: 16.3 -> 6.5, against eight warps that
// searched the references by four dependent shared-memory loads; 31 -> 27.5 us with a second group of epilogue warps.
constexpr int GD_NORM_REFS = 18;                               // -inf, up to 15 references, +inf, padded
struct NormTables {
    float ref[2][64][GD_NORM_REFS];
    float4 guess[2][64];                                       // inv, off: count ~ rint(top * sat((y - mu) / sqrt(V) * inv + off)); sign of the gain
    float2 step[64];                                           // i and RN(1/i)
};

__device__ __noinline__ uint32_t norm_count_all(const float* r, float ds, float V) {
    uint32_t cnt = 0;
    for (int t = 1; r[t] < INFINITY; ++t) cnt += ds > __fmul_rn(V, r[t]) ? 1u : 0u;
    return cnt;
}

template <bool SMALL, bool PACKED>
__device__ __forceinline__ void direct_norm_head(const GemmParams& P, const EpiParams& ep, int buf, uint32_t taddr, int tile_col,
                                                 const NormTables& nt, int seg, long long row, bool row_ok, int col) {
    float mu = 0.0f, S = 0.0f;
    // statistics, in channel order
#pragma unroll 1
    for (int c0 = 0; c0 < 64; c0 += 16) {
        uint32_t v[16];
        ptx::tmem_ld16(taddr + (uint32_t)c0, v);
        const float4* const pa = reinterpret_cast<const float4*>(&ep.a[buf][tile_col + c0]);
        const float4* const pb = reinterpret_cast<const float4*>(&ep.b[buf][tile_col + c0]);
        const float4* const ps = reinterpret_cast<const float4*>(&nt.step[c0]);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int i4 = 0; i4 < 4; ++i4) {
            const float4 a4 = pa[i4], b4 = pb[i4], s01 = ps[2 * i4], s23 = ps[2 * i4 + 1];
            float y[4];
            f2_unpack(f2_fma(acc_to_float2<SMALL, PACKED>(v[4 * i4], v[4 * i4 + 1], P.shift), f2_pack(a4.x, a4.y), f2_pack(b4.x, b4.y)), y[0], y[1]);
            f2_unpack(f2_fma(acc_to_float2<SMALL, PACKED>(v[4 * i4 + 2], v[4 * i4 + 3], P.shift), f2_pack(a4.z, a4.w), f2_pack(b4.z, b4.w)), y[2], y[3]);
            const float fi[4] = {s01.x, s01.z, s23.x, s23.z}, ri[4] = {s01.y, s01.w, s23.y, s23.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float delta = __fadd_rn(y[j], -mu);
                // RN(delta / i): quotient estimate, exact remainder in one FMA, one correction
                const float q0 = __fmul_rn(delta, ri[j]);
                const float rem = __fmaf_rn(-q0, fi[j], delta);
                mu = __fadd_rn(mu, __fmaf_rn(rem, ri[j], q0));
                S = __fadd_rn(S, __fmul_rn(delta, __fadd_rn(y[j], -mu)));
            }
        }
    }
    const float V = __fadd_rn(S, P.n_eps);
    if (P.norm_stats != nullptr && row_ok) {
        const int heads = P.norm_dim >> 6, head = (col - seg * P.norm_dim) >> 6;
        *reinterpret_cast<float2*>(P.norm_stats + ((long long)seg * P.M * heads + row * heads + head) * 2) = make_float2(mu, V);
    }
    // levels
    const f32x2 nmu2 = f2_dup(-mu), rs2 = f2_dup(rsqrtf(V)), V2 = f2_dup(V), top2 = f2_dup((float)((1 << P.norm_bits) - 1));
    uint8_t* o = (uint8_t*)P.out + row * P.ld_out + (((long long)col * P.out_c) >> 3);
    const uint32_t qn_low = ((uint32_t)P.norm_qn & 0x7Fu) * 0x01010101u, qn_top = ((uint32_t)P.norm_qn & 0x80u) * 0x01010101u;
    uint32_t ref0 = ptx::smem_addr(&nt.ref[seg][0][0]) - 0x4B400000u * 4u;         // the guess is 1.5*2^23 + count: times four an address
#pragma unroll 1
    for (int c0 = 0; c0 < 64; c0 += 16) {
        uint32_t v[16], w[4];
        ptx::tmem_ld16(taddr + (uint32_t)c0, v);
        const float4* const pa = reinterpret_cast<const float4*>(&ep.a[buf][tile_col + c0]);
        const float4* const pb = reinterpret_cast<const float4*>(&ep.b[buf][tile_col + c0]);
        const float4* const pg = &nt.guess[seg][c0];
        ptx::tmem_ld_wait();
#pragma unroll
        for (int i4 = 0; i4 < 4; ++i4) {
            const float4 a4 = pa[i4], b4 = pb[i4];
            float ds[4];
            uint32_t g[4];
            bool proven = true;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int i = 4 * i4 + 2 * p;
                const float4 ga = pg[i], gb = pg[i + 1];
                const f32x2 y = f2_fma(acc_to_float2<SMALL, PACKED>(v[i], v[i + 1], P.shift), p ? f2_pack(a4.z, a4.w) : f2_pack(a4.x, a4.y),
                                       p ? f2_pack(b4.z, b4.w) : f2_pack(b4.x, b4.y));
                const f32x2 delta = f2_add(y, nmu2), d = f2_mul(delta, f2_pack(ga.z, gb.z));             // exact sign change
                float d0, d1, q0, q1, u0, u1, g0, g1, l0, l1, h0, h1;
                f2_unpack(d, d0, d1);
                f2_unpack(f2_mul(d, d), q0, q1);
                ds[2 * p] = copysignf(q0, d0);
                ds[2 * p + 1] = copysignf(q1, d1);
                f2_unpack(f2_mul(delta, rs2), u0, u1);
                u0 = __saturatef(fmaf(u0, ga.x, ga.y));
                u1 = __saturatef(fmaf(u1, gb.x, gb.y));
                f2_unpack(f2_fma(f2_pack(u0, u1), top2, f2_dup(12582912.0f)), g0, g1);
                g[2 * p] = __float_as_uint(g0);
                g[2 * p + 1] = __float_as_uint(g1);
                const uint32_t r0 = g[2 * p] * 4u + ref0, r1 = g[2 * p + 1] * 4u + ref0;
                f2_unpack(f2_mul(V2, f2_pack(ptx::ld_shared_f32(r0 + 4 * i * GD_NORM_REFS), ptx::ld_shared_f32(r1 + 4 * (i + 1) * GD_NORM_REFS))), l0, l1);
                f2_unpack(f2_mul(V2, f2_pack(ptx::ld_shared_f32(r0 + 4 * (i * GD_NORM_REFS + 1)), ptx::ld_shared_f32(r1 + 4 * ((i + 1) * GD_NORM_REFS + 1)))), h0, h1);
                proven = proven && ds[2 * p] > l0 && !(ds[2 * p] > h0) && ds[2 * p + 1] > l1 && !(ds[2 * p + 1] > h1);
            }
            uint32_t n = (g[0] + (g[1] << 8) + (g[2] << 16) + (g[3] << 24)) - 0x4B400000u * 0x01010101u;
            if (!proven) {
                n = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) n |= norm_count_all(nt.ref[seg][c0 + 4 * i4 + j], ds[j], V) << (8 * j);
            }
            w[i4] = (n + qn_low) ^ qn_top;                      // Qn added to every byte (none overflows: low bits, then the top bit)
        }
        if (row_ok) {
            if (P.out_c == 8) {
                *reinterpret_cast<uint4*>(o) = make_uint4(w[0], w[1], w[2], w[3]);
            } else if (P.out_c == 4) {
                uint32_t t[2];
                narrow4(w, t);
                *reinterpret_cast<uint2*>(o) = make_uint2(t[0], t[1]);
            } else {
                *reinterpret_cast<uint32_t*>(o) = narrow2(w);
            }
        }
        o += 2 * P.out_c;
        ref0 += 4u * 16u * GD_NORM_REFS;
    }
}

// A tile's rows and columns.  The norm kind numbers its tiles by column first, Q and K before V, so that the cheap V tiles
// fill the last round, and no tile crosses from one of the three segments into the next.
template <int KIND>
__device__ __forceinline__ void direct_tile(const GemmParams& P, int tile, int& m_tile, int& col_t, int& cols) {
    if (KIND == EK_QKV_NORM) {
        const int n = tile / P.m_tiles, per_seg = P.n_tiles / 3;
        m_tile = tile - n * P.m_tiles;
        const int seg = n / per_seg, off = (n - seg * per_seg) * P.bn;
        col_t = seg * P.norm_dim + off;
        cols = P.norm_dim - off < P.bn ? P.norm_dim - off : P.bn;
    } else {
        m_tile = tile / P.n_tiles;
        col_t = (tile - m_tile * P.n_tiles) * P.bn;
        cols = P.N - col_t < P.bn ? P.N - col_t : P.bn;                       // whole blocks, but for the last tile of a ragged width
    }
}

// RAGGED: codes of a width that is no multiple of the column block.  A variant of its own: with the choice made at run time and the
// second tensor map passed to every launch, twelve layers on one image, none of them ragged, took 332 us instead of 328.
// GROUPS of epilogue warps.  The norm kind has two where CTAs have several tiles, each with an accumulator buffer of its own: a thread's
// walk through Eq. 5 is a chain, three warps a scheduler leave half of its slots empty, and a second tile beside the first fills
// them (12,672 x 384 -> 1152 31 -> 27.5 us).  Without a second tile 832 threads only start later than 448: 198 x 64 6.7 us with two
// groups, 6.2 with one.
template <int KIND, bool SMALL, bool RES, bool PACKED, bool RAGGED = false, int GROUPS = 1>
__global__ void __launch_bounds__(gd_threads(KIND, PACKED, GROUPS), 1)
gemm_direct_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                   const __grid_constant__ DirectExtra<KIND, RAGGED> X, const __grid_constant__ GemmParams P) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ DirectBars bars;
    __shared__ __align__(16) EpiParams epi_params_of[GROUPS];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) std::conditional_t<KIND == EK_QKV_NORM, NormTables, float4> norm_tab[1];
    constexpr int BLK = gd_block(KIND);
    constexpr int EPI_W = gd_epi_warps(KIND, PACKED), SLICES = EPI_W / 4;
    constexpr int WARP_TMA_D = gd_threads(KIND, PACKED, GROUPS) / 32 - 2, WARP_MMA_D = WARP_TMA_D + 1;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
    uint8_t* const smem_gen = smem_raw + (smem_base - ptx::smem_addr(smem_raw));
    const bool resident = PACKED && P.b_resident;
    const int ragged_col = (P.n_tiles - 1) * P.bn;             // (RAGGED) column of the tile that ends inside a column block
    const uint32_t stage_bytes = P.ia_bytes + (resident ? 0u : P.ib_bytes);
    const uint32_t packed_off = (uint32_t)P.ns_i * stage_bytes, stage_packed = P.pa_bytes + P.pb_bytes;     // packed operands' ring
    const uint32_t resident_off = packed_off + (uint32_t)P.ns_p * stage_packed;
    volatile int* abort_ptr = &abort_flag;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < MAX_STAGES; ++s) {
            ptx::mbar_init(ptx::smem_addr(&bars.full[s]), PACKED ? GD_UNPACK_WARPS / 2 + ((P.a_direct || P.b_direct) ? 1 : 0) : 1);
            ptx::mbar_init(ptx::smem_addr(&bars.empty[s]), 1);
            if (PACKED) {
                ptx::mbar_init(ptx::smem_addr(&bars.p_full[s]), 1);
                ptx::mbar_init(ptx::smem_addr(&bars.p_empty[s]), GD_UNPACK_WARPS / 2);
            }
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(ptx::smem_addr(&bars.acc_full[b]), 1);
            ptx::mbar_init(ptx::smem_addr(&bars.acc_empty[b]), EPI_W);
        }
        for (int k = 0; k < GROUPS; ++k) ptx::mbar_init(ptx::smem_addr(&bars.epi_sync[k]), EPI_W);
        ptx::fence_mbar_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == WARP_MMA_D) {
        ptx::tmem_alloc(ptx::smem_addr(&tmem_base_slot), P.tmem_cols);
        ptx::tmem_relinquish();
    }
    if (warp == WARP_TMA_D && lane == 0) {
        ptx::prefetch_tensormap(&map_a);
        ptx::prefetch_tensormap(&map_b);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, tmem_base_slot, 0);      // warp-uniform, as is `warp`
    const uint32_t acc_stride = P.tmem_cols >> 1;
    // Operands, parameters and the residual may come from the previous kernel.  Where weights and parameters cannot, the producer
    // fills the ring with weights, asks for the rest of the tile's into L2, and the epilogue fetches its first parameters before
    // it waits: at small batches they come from HBM, beside the previous kernel instead of behind it (with the gains of LayerNorm
    // and the exp table, twelve layers on one image 352 -> 326 us (now 321), a layer at batch 8 47.1 -> 45.1, 8 bits at batch 32 117.8 -> 114.8).
    const bool early = !PACKED && P.at_rest;
    auto dependency = [&]() {
        grid_dependency_wait();
        grid_dependency_launch();
    };
    if (!early) dependency();

    if (warp == WARP_TMA_D) {
        {
            // Weights of a tile: permuted within column blocks, or in their own order
            auto load_weights = [&](uint32_t dst, uint32_t bar, int byte, int col) {
                bool ordered = false;
                if constexpr (KIND == EK_QKV_NORM) ordered = col < 2 * P.norm_dim;
                else if constexpr (RAGGED) ordered = col >= ragged_col;
                if constexpr (KIND == EK_QKV_NORM || RAGGED)
                    if (ordered) { ptx::tma_load_4d(dst, &X.map_w, bar, byte, col, 0, 0); return; }
                ptx::tma_load_5d(dst, &map_b, bar, byte, 0, 0, 0, col / BLK);
            };
            // K blocks of the first tile that are on their way before the loop, which a test for them would slow down in every call
            // (12,608 x 384 -> 384 to fp32 7.0 -> 7.4 us)
            int loaded = 0;
            if (early) {
                int m_tile, col_t, cols;
                direct_tile<KIND>(P, blockIdx.x, m_tile, col_t, cols);
                loaded = P.k_blocks < P.ns_i ? P.k_blocks : P.ns_i;
                if (ptx::elect_one()) {
                    for (int kb = 0; kb < loaded; ++kb) {
                        const uint32_t bar = ptx::smem_addr(&bars.full[kb]);
                        ptx::mbar_arrive_expect_tx(bar, stage_bytes);
                        load_weights(smem_base + (uint32_t)kb * stage_bytes + P.ia_bytes, bar, kb * BK, col_t);
                    }
                    // (by the CTAs of the first row tiles: all row tiles share them)
                    if (m_tile < 2 && (!RAGGED || col_t < ragged_col))
                        for (int kb = loaded; kb < P.k_blocks; ++kb) ptx::tma_prefetch_5d(&map_b, kb * BK, 0, 0, 0, col_t / BLK);
                }
                __syncwarp();
                dependency();
                if (ptx::elect_one())
                    for (int kb = 0; kb < loaded; ++kb)
                        ptx::tma_load_4d(smem_base + (uint32_t)kb * stage_bytes, &map_a, ptx::smem_addr(&bars.full[kb]), kb * BK, m_tile * BM, 0, 0);
                __syncwarp();
            }
            VT_TRACER(tr, lane == 0 ? 0 : -1);
            VT_STAMP(tr, TT_START);
            const uint32_t full0 = ptx::smem_addr(&bars.full[0]), empty0 = ptx::smem_addr(&bars.empty[0]);
            const int k_blocks = P.k_blocks, ns = P.ns_i;
            const bool wrapped = loaded == ns;
            int s = wrapped ? 0 : loaded, it = loaded, sp = 0, kb0 = loaded;
            uint32_t ph = wrapped ? 0u : 1u, dst = smem_base + (uint32_t)s * stage_bytes, php = 1u;
            bool ok = true;
            const uint32_t direct_bytes = PACKED ? (P.a_direct ? P.ia_bytes : 0u) + (P.b_direct ? P.ib_bytes : 0u) : stage_bytes;
            const int a_step = P.a_direct ? BK : 16 * P.ca, b_step = P.b_direct ? BK : 16 * P.cb;         // bytes of a row per K block
            for (int tile = blockIdx.x; ok && tile < P.total_tiles; tile += gridDim.x) {
                int m_tile, col_t, cols;
                direct_tile<KIND>(P, tile, m_tile, col_t, cols);
                const int m0 = m_tile * BM;
                for (int kb = kb0; kb < k_blocks; ++kb, ++it) {
                    const uint32_t full = full0 + 8u * (uint32_t)s;
                    uint32_t a_dst = dst, b_dst = dst + P.ia_bytes, a_bar = full, b_bar = full;
                    if (PACKED) {
                        if (!mbar_wait_warp(ptx::smem_addr(&bars.p_empty[sp]), php, abort_ptr)) { ok = false; break; }
                        const uint32_t p_full = ptx::smem_addr(&bars.p_full[sp]), p_dst = smem_base + packed_off + (uint32_t)sp * stage_packed;
                        if (ptx::elect_one()) ptx::mbar_arrive_expect_tx(p_full, resident && tile != (int)blockIdx.x ? P.pa_bytes : stage_packed);
                        if (!P.a_direct) { a_dst = p_dst; a_bar = p_full; }
                        if (!P.b_direct) { b_dst = p_dst + P.pa_bytes; b_bar = p_full; }
                        if (++sp == P.ns_p) { sp = 0; php ^= 1u; }
                    }
                    if (!PACKED || direct_bytes) {
                        VT_STAMP(tr, TT_WAIT_EMPTY);
                        if (!mbar_wait_warp(empty0 + 8u * (uint32_t)s, ph, abort_ptr)) { ok = false; break; }
                        VT_STAMP(tr, TT_GOT_EMPTY);
                        if (ptx::elect_one()) ptx::mbar_arrive_expect_tx(full, direct_bytes);
                    }
                    __syncwarp();
                    if (ptx::elect_one()) {
                        ptx::tma_load_4d(a_dst, &map_a, a_bar, kb * a_step, m0, 0, 0);
                        if (!resident || tile == (int)blockIdx.x) load_weights(b_dst, b_bar, kb * b_step, col_t);
                    }
                    __syncwarp();
                    if (++s == ns) { s = 0; ph ^= 1u; dst = smem_base; } else dst += stage_bytes;
                }
                kb0 = 0;
            }
            if (!ok) {
                // give the copies still in flight a bounded chance to land before the CTA exits
                for (int j = (it > MAX_STAGES ? it - MAX_STAGES : 0); j <= it; ++j) {
                    if (PACKED && j + P.ns_p > it) {
                        const uint32_t bar = ptx::smem_addr(&bars.p_full[j % P.ns_p]);
                        for (int spin = 0; spin < (1 << 20) && !ptx::mbar_try_wait(bar, (uint32_t)(j / P.ns_p) & 1u); ++spin) {}
                    }
                    if (direct_bytes && j + ns > it) {
                        const uint32_t bar = full0 + 8u * (uint32_t)(j % ns);
                        for (int spin = 0; spin < (1 << 20) && !ptx::mbar_try_wait(bar, (uint32_t)(j / ns) & 1u); ++spin) {}
                    }
                }
            }
        }
    } else if (warp == WARP_MMA_D) {
        {
            if (early) dependency();
            const uint32_t idesc = ptx::idesc_i8(BM, P.bn, P.a_signed, P.b_signed, 0);
            VT_TRACER(tr, lane == 0 ? 1 : -1);
            VT_STAMP(tr, TT_START);
            const uint64_t a_desc0 = ptx::smem_desc(smem_base, 16, 1024, ptx::SWIZZLE_128B);
            const uint64_t b_desc0 = ptx::smem_desc(smem_base + (resident ? resident_off : P.ia_bytes), 16, 1024, ptx::SWIZZLE_128B);
            const uint64_t stage_step = (uint64_t)(stage_bytes >> 4);        // descriptor address field counts 16-byte units
            const uint32_t full0 = ptx::smem_addr(&bars.full[0]), empty0 = ptx::smem_addr(&bars.empty[0]);
            const int k_blocks = P.k_blocks, ns = P.ns_i;
            // MMAs of the last (possibly partial) K block; 64 two-bit codes share a chunk, whose reordered codes fill two steps
            int last_steps = (P.K - (k_blocks - 1) * BK + 31) / 32;
            if (PACKED && P.reorder && P.ca == 2) last_steps = (last_steps + 1) & ~1;
            int s = 0, tl = 0;
            uint32_t ph = 0;
            uint64_t a_desc = a_desc0, b_desc = b_desc0;
            bool ok = true;
            for (int tile = blockIdx.x; ok && tile < P.total_tiles; tile += gridDim.x, ++tl) {
                const int buf = tl & 1;
                const uint32_t acc_ph = (uint32_t)(tl >> 1) & 1u;
                VT_STAMP(tr, TT_WAIT_EMPTY);
                if (!mbar_wait_warp(ptx::smem_addr(&bars.acc_empty[buf]), acc_ph ^ 1u, abort_ptr)) { ok = false; break; }
                VT_STAMP(tr, TT_GOT_EMPTY);
                ptx::tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)buf * acc_stride;
                if (resident) b_desc = b_desc0;
                for (int kb = 0; kb < k_blocks; ++kb) {
                    VT_STAMP(tr, TT_WAIT_FULL);
                    if (!mbar_wait_warp(full0 + 8u * (uint32_t)s, ph, abort_ptr)) { ok = false; break; }
                    VT_STAMP(tr, TT_GOT_FULL);
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
                        if (kb + 1 < k_blocks || last_steps == 4) {              // 32 int8 of K per MMA: 32 bytes along a swizzled row
                            ptx::mma_i8(d_tmem, a_desc, b_desc, idesc, kb != 0 ? 1u : 0u);
                            ptx::mma_i8(d_tmem, a_desc + 2u, b_desc + 2u, idesc, 1u);
                            ptx::mma_i8(d_tmem, a_desc + 4u, b_desc + 4u, idesc, 1u);
                            ptx::mma_i8(d_tmem, a_desc + 6u, b_desc + 6u, idesc, 1u);
                        } else {
                            for (int k = 0; k < last_steps; ++k)
                                ptx::mma_i8(d_tmem, a_desc + (uint64_t)(k * 2), b_desc + (uint64_t)(k * 2), idesc, (kb | k) != 0 ? 1u : 0u);
                        }
                        ptx::mma_commit(empty0 + 8u * (uint32_t)s);
                    }
                    __syncwarp();
                    if (resident) b_desc += (uint64_t)(P.ib_bytes >> 4);
                    if (++s == ns) { s = 0; ph ^= 1u; a_desc = a_desc0; if (!resident) b_desc = b_desc0; }
                    else { a_desc += stage_step; if (!resident) b_desc += stage_step; }
                }
                if (ok && ptx::elect_one()) ptx::mma_commit(ptx::smem_addr(&bars.acc_full[buf]));
                VT_STAMP(tr, TT_ISSUED);
            }
        }
    } else if (PACKED && warp >= EPI_W) {
        // Packed codes -> int8 operand tiles: 48 KB for a K block of a 128 x 256 tile.  Two groups of four warps take K blocks
        // in turn, so that one group's waits, shared-memory latency and proxy fence run beside the other's work.
        const int grp = (warp - EPI_W) >> 2, tid_u = threadIdx.x - (EPI_W + 4 * grp) * 32;
        const int ns = P.ns_i, ns_p = P.ns_p;
        int s = grp % ns, sp = grp % ns_p;
        uint32_t ph = 1u, php = 0u;
        bool ok = true;
        int kb = grp, tile = blockIdx.x;
        while (kb >= P.k_blocks) { kb -= P.k_blocks; tile += gridDim.x; }
        while (ok && tile < P.total_tiles) {
            // The operand slot first: a parity tells a phase only from the one before it, and the phase of p_full[sp] before this
            // block's is block it - ns_p, the other group's where ns_p is odd.  Once block it - ns has been contracted (blocks are
            // contracted in order) every block up to it has landed, it - ns_p among them unless ns_p = 2 < ns, where that one is
            // this group's own.  Asked first, the packed slot could answer for block it - 3 of a ring of three before that block
            // had landed, and the old bytes would be expanded.
            bool w = mbar_wait(ptx::smem_addr(&bars.empty[s]), ph, abort_ptr);
            w = w && mbar_wait(ptx::smem_addr(&bars.p_full[sp]), php, abort_ptr);
            if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
            ptx::tc_fence_after();
            const uint8_t* pa = smem_gen + packed_off + (size_t)sp * stage_packed;
            uint8_t* ia = smem_gen + (size_t)s * stage_bytes;
            if (!P.a_direct) direct_unpack(P.ca, P.a_signed, P.reorder, pa, ia, BM, tid_u);
            if (!P.b_direct && (!resident || tile == (int)blockIdx.x))
                direct_unpack(P.cb, P.b_signed, P.reorder, pa + P.pa_bytes, resident ? smem_gen + resident_off + (size_t)kb * P.ib_bytes : ia + P.ia_bytes,
                              P.bn, tid_u);
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(ptx::smem_addr(&bars.full[s]));
                ptx::mbar_arrive(ptx::smem_addr(&bars.p_empty[sp]));
            }
            if ((s += 2) >= ns) { s -= ns; ph ^= 1u; }
            if ((sp += 2) >= ns_p) { sp -= ns_p; php ^= 1u; }
            kb += 2;
            while (kb >= P.k_blocks) { kb -= P.k_blocks; tile += gridDim.x; }
        }
    } else {
        const int grp = GROUPS == 1 ? 0 : warp / EPI_W;                        // takes every GROUPS-th tile of the CTA
        const int q4 = warp & 3, slice = (warp - grp * EPI_W) >> 2;
        const int tid_e = threadIdx.x - grp * EPI_W * 32;
        const int first_tile = (int)blockIdx.x + grp * (int)gridDim.x, tile_step = GROUPS * (int)gridDim.x;
        EpiParams& epi_params = epi_params_of[grp];
        const uint32_t epi_sync = ptx::smem_addr(&bars.epi_sync[grp]);
        const float down = __int_as_float((127 - (SMALL ? 0 : P.shift)) << 23);
        // per-column parameters of a tile (multiplier, bias, GELU output factor), column c of the tile
        auto fetch_params = [&](int tile, int c, float& a, float& b, float& q) {
            int m_tile, col_t, cols;
            direct_tile<KIND>(P, tile, m_tile, col_t, cols);
            const int n = col_t + c;
            a = 0.0f; b = 0.0f; q = 0.0f;
            if (c < cols) {
                if (KIND == EK_REQUANT) {
                    a = __ldg(P.col_a + n);
                } else if (KIND == EK_QKV_NORM && col_t >= 2 * P.norm_dim) {   // V: folded requantization
                    a = __ldg(P.v_alpha + (n - 2 * P.norm_dim));
                } else {
                    a = P.col_a ? __fmul_rn(P.x_step, __ldg(P.col_a + n)) : P.x_step;
                    if (KIND == EK_REQUANT_GELU) q = __fdiv_rn(0.5f * __ldg(P.inv_s + n), P.out_qp);   // folds GELU's 1/2 and 1/Qp
                }
                if (KIND == EK_QKV_NORM && col_t >= 2 * P.norm_dim) b = P.v_beta ? __ldg(P.v_beta + (n - 2 * P.norm_dim)) : 0.0f;
                else b = P.col_b ? __ldg(P.col_b + n) : 0.0f;
                if (PACKED) a *= down;
            }
        };
        // The parameters of tile i+1 are fetched while the warps wait for tile i's accumulators and are stored to the other
        // half of epi_params before tile i is processed, so no tile waits for them.  (bn <= 256 <= epilogue threads)
        const bool my_col = tid_e < P.bn;
        auto put_params = [&](int tile, int buf, float a, float b, float q) {
            int my_slot = gd_param_slot<BLK>(tid_e);
            if (KIND == EK_QKV_NORM) {
                int m_tile, col_t, cols;
                direct_tile<KIND>(P, tile, m_tile, col_t, cols);
                if (col_t < 2 * P.norm_dim) my_slot = tid_e;                  // Q and K: columns in order
            } else if (RAGGED) {
                int m_tile, col_t, cols;
                direct_tile<KIND>(P, tile, m_tile, col_t, cols);
                if (col_t >= ragged_col) my_slot = tid_e;
            }
            epi_params.a[buf][my_slot] = a;
            epi_params.b[buf][my_slot] = b;
            if (KIND == EK_REQUANT_GELU) epi_params.q[buf][my_slot] = q;
        };
        if (my_col && first_tile < P.total_tiles) {
            float a, b, q;
            fetch_params(first_tile, tid_e, a, b, q);
            put_params(first_tile, 0, a, b, q);
        }
        if (early) dependency();
        if (KIND == EK_REQUANT && P.exp_table != nullptr)
            fill_exp_table(P.exp_table, P.exp_smax, P.exp_c, blockIdx.x * (EPI_W * 32) + tid_e, gridDim.x * (EPI_W * 32));
        int tl = 0;
        bool ok = true;
        VT_TRACER(tr, (lane == 0 && warp == 0) ? 2 : ((lane == 0 && warp == EPI_W - 1) ? 3 : -1));
        VT_STAMP(tr, TT_START);
        // fp32 kinds: the residual of the warp's next two units of 16 rows x 32 columns, requested two units ahead across tiles
        float res[2][2][8];
        int ahead_tile = first_tile, ahead_u = slice;
        auto request_residual = [&](float (&r)[2][8]) {
            for (; ahead_tile < P.total_tiles; ahead_tile += tile_step, ahead_u = slice) {
                int m_tile, col_t, cols;
                direct_tile<KIND>(P, ahead_tile, m_tile, col_t, cols);
                if ((ahead_u >> 1) * BLK < cols) {
                    const int row0 = m_tile * BM + q4 * 32 + 16 * (ahead_u & 1);
                    direct_residual(P, lane, row0, P.M - row0, col_t + (ahead_u >> 1) * BLK, r);
                    ahead_u += SLICES;
                    break;
                }
            }
        };
        if constexpr (KIND == EK_QKV_NORM) {
            // laid out once for all groups, which meet before any of them reads it
            const int nt = (1 << P.norm_bits) - 1;
            for (int i = threadIdx.x; i < 2 * 64; i += GROUPS * EPI_W * 32) {
                const int set = i >> 6, c = i & 63;
                const float* r = P.norm_refs + (size_t)i * nt;
                float* const dst = norm_tab[0].ref[set][c];
                dst[0] = -INFINITY;
                for (int t = 0; t < GD_NORM_REFS - 1; ++t) dst[t + 1] = t < nt ? __ldg(r + t) : INFINITY;
                const float r0 = __ldg(r), r1 = __ldg(r + nt - 1), sgn = (P.norm_flip != nullptr && __ldg(P.norm_flip + i)) ? -1.0f : 1.0f;
                const float rho0 = copysignf(sqrtf(fabsf(r0)), r0), rho1 = copysignf(sqrtf(fabsf(r1)), r1);
                float inv = (float)(nt - 1) / (rho1 - rho0);
                if (!(inv < 1e30f)) inv = 0.0f;
                norm_tab[0].guess[set][c] = make_float4(inv * sgn / (float)nt, (0.5f - rho0 * inv) / (float)nt, sgn, 0.0f);
                if (set == 0) norm_tab[0].step[c] = make_float2((float)(c + 1), __frcp_rn((float)(c + 1)));
            }
            if constexpr (GROUPS > 1) asm volatile("bar.sync 1, %0;" ::"n"(GROUPS * EPI_W * 32) : "memory");
        }
        if (KIND == EK_DEQUANT && RES) {
            request_residual(res[0]);
            request_residual(res[1]);
        }
        for (int tile = first_tile; ok && tile < P.total_tiles; tile += tile_step, ++tl) {
            int m_tile, col_t, cols;
            direct_tile<KIND>(P, tile, m_tile, col_t, cols);
            const int buf = tl & 1;                                            // half of the parameters
            const int acc = GROUPS == 1 ? buf : grp;                           // accumulator buffer
            const int next_tile = tile + tile_step;
            const bool fetch_next = my_col && next_tile < P.total_tiles;
            float na = 0.0f, nb = 0.0f, nq = 0.0f;
            if (fetch_next) fetch_params(next_tile, tid_e, na, nb, nq);
            const int row_q = m_tile * BM + q4 * 32;
            const int rows_q = P.M - row_q;                                   // valid rows from the quarter's first one on
            const uint32_t acc_ph = (uint32_t)(GROUPS == 1 ? tl >> 1 : tl) & 1u;
            VT_STAMP(tr, TT_WAIT_ACC);
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(epi_sync);
            bool w = mbar_wait(epi_sync, (uint32_t)tl & 1u, abort_ptr);
            VT_STAMP(tr, TT_WAIT_FULL);
            w = w && mbar_wait(ptx::smem_addr(&bars.acc_full[acc]), acc_ph, abort_ptr);
            VT_STAMP(tr, TT_GOT_ACC);
            if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
            ptx::tc_fence_after();
            if (fetch_next) put_params(next_tile, buf ^ 1, na, nb, nq);                  // every warp has passed the barrier: none reads that half
            const uint32_t t_quarter = tmem_base + (uint32_t)acc * acc_stride + ((uint32_t)(q4 * 32) << 16);
            const int n_blk = cols / BLK;
            if constexpr (KIND == EK_DEQUANT) {
                // Units of half a block: 192 columns are three for every slice, where whole blocks were two for half of the slices
                // (25,344 x 384 -> 384: 19.0 -> 17.4 us, 12,608 x 768 -> 768: 20.0 -> 18.6)
                auto unit = [&](int u, const float (&r)[2][8]) {
                    uint32_t v[16];
                    const int blk = u >> 1, half = u & 1;
                    ptx::tmem_ld_frag32(t_quarter + ((uint32_t)half << 20) + (uint32_t)(blk * BLK), v);
                    ptx::tmem_ld_wait();
                    direct_f32<SMALL, RES, PACKED>(P, v, epi_params, buf, blk * BLK, lane, row_q + 16 * half, rows_q - 16 * half, col_t + blk * BLK, r);
                };
#pragma unroll 1
                for (int u = slice; u < 2 * n_blk; u += 2 * SLICES) {
                    unit(u, res[0]);
                    if (u + SLICES < 2 * n_blk) {
                        if (RES) request_residual(res[0]);
                        unit(u + SLICES, res[1]);
                    } else if (RES) {                                         // an odd number: the next tile starts with the other half
#pragma unroll
                        for (int i = 0; i < 16; ++i) res[0][i >> 3][i & 7] = res[1][i >> 3][i & 7];
                    }
                    if (RES) request_residual(res[1]);
                }
            } else {
                bool norm = false;                                            // the tile's weights are in their own order
                if constexpr (KIND == EK_QKV_NORM) {
                    norm = col_t < 2 * P.norm_dim;                            // a Q or K tile
#pragma unroll 1
                    for (int blk = slice; norm && blk < n_blk; blk += SLICES)
                        direct_norm_head<SMALL, PACKED>(P, epi_params, buf, t_quarter + (uint32_t)(blk * 64), blk * 64, norm_tab[0],
                                                        col_t >= P.norm_dim ? 1 : 0, row_q + lane, lane < rows_q, col_t + blk * 64);
                }
                constexpr int CK = KIND == EK_QKV_NORM ? EK_REQUANT : KIND;
                if constexpr (RAGGED) {
                    norm = col_t >= ragged_col;                               // not walked by blocks either
#pragma unroll 1
                    for (int c = 16 * slice; norm && c < cols; c += 16 * SLICES)
                        direct_codes_row<CK, SMALL, PACKED>(P, t_quarter + (uint32_t)c, epi_params, buf, c, row_q + lane, lane < rows_q, col_t + c);
                }
                // One 16-row half of a block at a time: 90 registers, so that sixteen warps fit.  (Eight warps that keep the
                // parameters of a block for both halves and read the next accumulators ahead: fc1 79 us against 72.)
#pragma unroll 1
                for (int u = slice; !norm && u < 2 * n_blk; u += SLICES) {
                    const int half = u & 1, tile_col = (u >> 1) * BLK;
                    uint32_t v[32];
                    ptx::tmem_ld_frag64(t_quarter + ((uint32_t)half << 20) + (uint32_t)tile_col, v);
                    CodeParams<CK == EK_REQUANT_GELU> cp;
                    cp.load(epi_params, buf, tile_col, lane);
                    ptx::tmem_ld_wait();
                    direct_codes<CK, SMALL, PACKED>(P, v, cp, lane, row_q + 16 * half, rows_q - 16 * half, col_t + tile_col);
                }
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&bars.acc_empty[acc]));
            VT_STAMP(tr, TT_TILE_DONE);
        }
        VT_STAMP(tr, TT_END);
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA_D) {
        ptx::tc_fence_after();
        __syncwarp();
        ptx::tmem_dealloc(tmem_base, P.tmem_cols);
    }
}

// The weight matrix as the five-dimensional view whose tile copy lands permuted within blocks of `block` rows:
// (byte, e, q, g, block) with row = block * B + (B/4) q + 2g + e.
int make_map_permuted(CUtensorMap* map, const void* base, uint64_t row_bytes, uint64_t rows, uint64_t pitch, int block, int bn,
                      int container) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return VITINT_ERR_CUDA;
    const cuuint64_t g = (cuuint64_t)block / 8;
    cuuint64_t dims[5] = {row_bytes, 2, 4, g, rows / (uint64_t)block};
    cuuint64_t strides[4] = {pitch, pitch * (uint64_t)(block / 4), pitch * 2, pitch * (uint64_t)block};
    cuuint32_t box[5] = {(cuuint32_t)(16 * container), 2, 4, (cuuint32_t)g, (cuuint32_t)(bn / block)};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 5, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, container == 8 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? VITINT_OK : VITINT_ERR_CUDA;
}

// Which calls this kernel takes: codes of at least a column block, fp32 outputs of whole column blocks whose rows, and the residual's,
// lie on 32 bytes, no batch of problems.  Everything else stays with gemm_i8_kernel.
bool direct_eligible(const GemmParams& P, int n_inner, int n_outer, int b_mn_major) {
    if (n_inner != 1 || n_outer != 1 || b_mn_major) return false;
    if (P.kind == EK_QKV_NORM) return true;
    if (P.kind == EK_REQUANT || (P.kind == EK_REQUANT_GELU && P.unit_out)) {
        // A ragged width takes a second tensor map, 0.4 us of the host's time, which a small call waits for longer than for the GPU
        // (with a quantizer in front, 1015 x 320 -> 1290 14.0 / 14.7 us, 197 x 768 -> 1000 14.1 / 14.8) unless it is recorded; larger
        // ones gain: 12,608 x 768 -> 1290 33.9 -> 29.4 us, 50,000 x 256 -> 70 22.4 -> 20.9, recorded 1015 x 320 -> 1290 6.8 -> 4.4.
        return P.N % 64 == 0 || (P.N >= 64 && (launches_recorded() || (long long)P.M * P.N * P.K > 800ll * 1000 * 1000));
    }
    if (P.kind != EK_DEQUANT || P.N % 32 != 0) return false;
    // A short contraction whose residual and output exceed L2 is bound by HBM, and gemm_i8_kernel's asynchronous copies of the
    // residual through shared memory keep more of it in flight.  This kernel against that one, rotating buffers, residual and
    // output together: 50 MB 15.9 / 19.4, 15.6 / 16.6 and 15.4 / 20.5 us (K = N = 768, 384, 1024), 95 MB 27.1 / 27.1, 26.5 / 29.5 and
    // 26.7 / 29.0, 140 MB 37.2 / 34.5, 36.9 / 36.4 and 37.8 / 37.3, 400 MB 100 / 85, 100 / 95 and 100 / 93 (K = N = 192, two K
    // blocks: 15.6 / 15.6, 29.4 / 27.5, 37.6 / 32.5, 98 / 81).
    if (P.a_direct && P.b_direct && P.residual && P.K <= 1024 && (long long)P.M * P.N * 8 > 100ll * 1000 * 1000) return false;
    auto rows32 = [](const void* p, long long ld) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0 && ld % 8 == 0; };
    return rows32(P.out, P.ld_out) && (!P.residual || rows32(P.residual, P.ld_res));
}

// Tile width: the multiple of the column block with the least estimated time
//     fill (K blocks x 0.17 us) + (waves - 1) x max(K blocks x max(0.17, 0.00125 columns) us, epilogue) + epilogue
// where the epilogue takes 0.55 us and 8 ns a column (requantize), 0.85 and 12.4 (GELU) or 0.8 and 15.5 (fp32), as measured at
// M = 197 .. 25,344 and widths 32 .. 256: below 136 columns a K block costs the same at every width, so a grid that does not
// fill the chip takes narrow tiles (197 x 768 x 768 fp32: 7.1 us at 256 columns, 3.6 at 32) and a full one the widest that does
// not add a wave (25,344 x 384 -> 1152: 20.9 us at 192 columns in nine waves, 19.3 at 256 in seven; 6304 x 768 -> 768 fp32:
// 10.0 at 192, 9.4 at 160, both two waves).
int direct_tile_columns(const GemmParams& P) {
    const int block = gd_block(P.kind), sms = sm_count();
    const int segments = P.kind == EK_QKV_NORM ? 3 : 1, width = P.N / segments;
    const float per_col = P.kind == EK_QKV_NORM ? 0.017f : P.kind == EK_REQUANT ? 0.008f : P.kind == EK_DEQUANT ? 0.0155f : 0.0124f;
    const float per_tile = P.kind == EK_QKV_NORM ? 0.2f : P.kind == EK_REQUANT ? 0.55f : P.kind == EK_DEQUANT ? 0.8f : 0.85f;
    int best = 0;
    float best_t = 0.0f;
    for (int bn = P.kind == EK_QKV_NORM ? 192 : MAX_BN; bn >= block; bn -= block) {
        if (bn > width && bn - block >= width) continue;
        const long long tiles = (long long)P.m_tiles * ((width + bn - 1) / bn) * segments;
        const float waves = (float)((tiles + sms - 1) / sms), epi = per_tile + per_col * (float)bn;
        const float k_main = (float)P.k_blocks * (bn > 136 ? 0.00125f * (float)bn : 0.17f);
        const float t = 0.17f * (float)P.k_blocks + (waves - 1.0f) * (k_main > epi ? k_main : epi) + epi;
        if (!best || t < best_t) { best = bn; best_t = t; }
    }
    return best;
}

int launch_gemm_direct(const CUtensorMap& map_a, const void* w, uint64_t w_row_bytes, uint64_t w_pitch, GemmParams P,
                       cudaStream_t st) {
    const int block = gd_block(P.kind);
    const bool packed = !P.a_direct || !P.b_direct;
    const bool alike = !P.a_direct && !P.b_direct && P.ca == P.cb;
    P.bn = direct_tile_columns(P);
    const int resident_bn = alike && P.kind != EK_QKV_NORM
        ? resident_tile_columns(sm_count(), P.m_tiles, P.k_blocks, P.N, P.cb, block, P.bn,
                                P.kind == EK_DEQUANT ? PE_FP32 : P.kind == EK_REQUANT ? PE_REQUANT : PE_GELU) : 0;
    P.b_resident = resident_bn != 0;
    if (resident_bn) P.bn = resident_bn;
    P.n_tiles = P.kind == EK_QKV_NORM ? 3 * ((P.norm_dim + P.bn - 1) / P.bn) : (P.N + P.bn - 1) / P.bn;
    const long long tiles = (long long)P.m_tiles * P.n_tiles;
    if (tiles > 0x7fffffffll) return VITINT_ERR_UNSUPPORTED;
    P.total_tiles = (int)tiles;
    P.ib_bytes = (uint32_t)P.bn * BK;
    P.pb_bytes = P.b_direct ? 0u : (uint32_t)P.bn * 16u * (uint32_t)P.cb;
    const uint32_t kept = P.b_resident ? (uint32_t)P.k_blocks * P.ib_bytes : 0u;       // (the plan keeps it below GD_RESIDENT_BYTES)
    const uint32_t stage = P.ia_bytes + (P.b_resident ? 0u : P.ib_bytes), stage_p = P.pa_bytes + P.pb_bytes;
    const uint32_t ring = P.b_resident ? GD_RESIDENT_BYTES - kept : GD_RING_BYTES - (P.kind == EK_QKV_NORM ? 8u * 1024u : 0u);     // beside 12 KB of static reference tables
    int ns, ns_p = 0;
    if (packed) {
        P.reorder = alike;
        ns = 3;
        while (ns > 2 && (uint32_t)ns * stage + 2u * stage_p > ring) --ns;
        ns_p = (int)((ring - (uint32_t)ns * stage) / stage_p);
        if (ns_p > MAX_STAGES) ns_p = MAX_STAGES;
    } else {
        ns = (int)(ring / stage);
        if (ns > MAX_STAGES) ns = MAX_STAGES;
    }
    P.ns_i = ns;
    P.ns_p = ns_p;
    const bool ragged = P.kind != EK_QKV_NORM && P.N % block != 0;
    P.at_rest = !packed && P.kind != EK_QKV_NORM && parameters_at_rest();
    uint32_t cols = 32;
    while (cols < 2u * (uint32_t)P.bn) cols <<= 1;
    P.tmem_cols = cols;
    CUtensorMap map_b;
    if (int rc = make_map_permuted(&map_b, w, w_row_bytes, (uint64_t)P.N, w_pitch, block, P.bn, P.b_direct ? 8 : P.cb)) return rc;
    size_t smem = (size_t)ns * stage + (size_t)ns_p * stage_p + kept + 1024;
    if (smem < 120 * 1024) smem = 120 * 1024;                  // two CTAs never share an SM (and its tensor memory)
    int grid = sm_count();
    if (P.b_resident) grid = grid / P.n_tiles * P.n_tiles;     // tile + grid lies in the same column of tiles
    if (grid > P.total_tiles) grid = P.total_tiles;
#ifdef VITINT_TRACE
    if (g_trace_max_ctas > 0 && grid > g_trace_max_ctas && !P.b_resident) grid = g_trace_max_ctas;
#endif
    const int dev = current_device();
    if (dev < 0) return VITINT_ERR_CUDA;
    static bool attr_set[MAX_DEVICES][30] = {};
    const int groups = P.kind == EK_QKV_NORM && !packed && P.total_tiles > grid ? 2 : 1;
    const int threads = gd_threads(P.kind, packed, groups);
    auto launch_with = [&](auto kernel, int slot, const auto& extra) -> int {
        if (!attr_set[dev][slot]) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(P.kind == EK_QKV_NORM || !packed ? GD_RING_BYTES : GD_RESIDENT_BYTES) + 1024) != cudaSuccess)
                return VITINT_ERR_CUDA;
            attr_set[dev][slot] = true;
        }
        launch_kernel(kernel, dim3(grid), dim3(threads), smem, st, map_a, map_b, extra, P);
        return cuda_status(cudaGetLastError());
    };
    auto launch = [&](auto kernel, int slot) -> int { return launch_with(kernel, slot, NoExtra{}); };
    auto by_operands = [&](auto small) -> int {
        constexpr bool S = decltype(small)::value;
        constexpr int s0 = S ? 0 : 15;
        if (P.kind == EK_DEQUANT) {
            if (packed) return P.residual ? launch(gemm_direct_kernel<EK_DEQUANT, S, true, true>, s0) : launch(gemm_direct_kernel<EK_DEQUANT, S, false, true>, s0 + 1);
            return P.residual ? launch(gemm_direct_kernel<EK_DEQUANT, S, true, false>, s0 + 2) : launch(gemm_direct_kernel<EK_DEQUANT, S, false, false>, s0 + 3);
        }
        if (P.kind == EK_QKV_NORM || ragged) {
            OrderExtra extra;
            if (int rc = make_map(&extra.map_w, w, w_row_bytes, (uint64_t)P.N, 1, 1, w_pitch, w_pitch * P.N, w_pitch * P.N,
                                  P.b_direct ? (uint32_t)BK : 16u * P.cb, (uint32_t)P.bn, P.b_direct != 0))
                return rc;
            if (P.kind == EK_QKV_NORM)
                return packed        ? launch_with(gemm_direct_kernel<EK_QKV_NORM, S, false, true>, s0 + 8, extra)
                       : groups == 2 ? launch_with(gemm_direct_kernel<EK_QKV_NORM, S, false, false, false, 2>, s0 + 9, extra)
                                     : launch_with(gemm_direct_kernel<EK_QKV_NORM, S, false, false>, s0 + 14, extra);
            if (P.kind == EK_REQUANT)
                return packed ? launch_with(gemm_direct_kernel<EK_REQUANT, S, false, true, true>, s0 + 10, extra)
                              : launch_with(gemm_direct_kernel<EK_REQUANT, S, false, false, true>, s0 + 11, extra);
            return packed ? launch_with(gemm_direct_kernel<EK_REQUANT_GELU, S, false, true, true>, s0 + 12, extra)
                          : launch_with(gemm_direct_kernel<EK_REQUANT_GELU, S, false, false, true>, s0 + 13, extra);
        }
        if (P.kind == EK_REQUANT) return packed ? launch(gemm_direct_kernel<EK_REQUANT, S, false, true>, s0 + 4) : launch(gemm_direct_kernel<EK_REQUANT, S, false, false>, s0 + 5);
        return packed ? launch(gemm_direct_kernel<EK_REQUANT_GELU, S, false, true>, s0 + 6) : launch(gemm_direct_kernel<EK_REQUANT_GELU, S, false, false>, s0 + 7);
    };
    return P.small_acc ? by_operands(std::true_type{}) : by_operands(std::false_type{});
}

}  // namespace
}  // namespace vitint

// Device helpers shared by the tensor-core kernels: the bounded mbarrier wait and the
// expansion of packed low-bit codes into int8 operand chunks.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace vitint {

constexpr long long WAIT_LIMIT_CYCLES = 2000000000ll;   // about one second

// Bounded wait.  Gives up after WAIT_LIMIT_CYCLES or as soon as another thread of the CTA
// has given up; the first to give up records the timeout in the device status word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          long long limit_cycles = WAIT_LIMIT_CYCLES) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        // sleeps in hardware until the phase completes or ~50 us pass, so a waiting warp leaves the
        // issue slots to the warps that have work
        if (ptx::mbar_try_wait_hint(bar, parity, 50000u)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit_cycles) {
            *abort_flag = 1;
            atomicExch(&g_device_status, (int)VITINT_ERR_TIMEOUT);
            return false;
        }
    }
}

// The same for a whole converged warp; the answer is warp-uniform.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}

// exp(fl32(s * c)) for every integer score s = -smax .. smax, correctly rounded to fp32 (fp64 exp, one rounding); thread `first` of
// `threads` that share the table.
__device__ __forceinline__ void fill_exp_table(float* table, int smax, float c, int first, int threads) {
    for (int i = first; i <= 2 * smax; i += threads) table[i] = (float)exp((double)__fmul_rn((float)(i - smax), c));
}

// 8 four-bit codes of one word -> 8 bytes in natural order.
template <int SGN>
__device__ __forceinline__ void unpack4(uint32_t w, uint32_t& o0, uint32_t& o1) {
    uint32_t lo, hi;
    if (SGN) { lo = (w << 4) & 0xF0F0F0F0u; hi = w & 0xF0F0F0F0u; }
    else     { lo = w & 0x0F0F0F0Fu;        hi = (w >> 4) & 0x0F0F0F0Fu; }
    o0 = __byte_perm(lo, hi, 0x5140);
    o1 = __byte_perm(lo, hi, 0x7362);
}
// 16 two-bit codes of one word -> 16 bytes in natural order.
template <int SGN>
__device__ __forceinline__ uint4 unpack2(uint32_t w) {
    uint32_t p0, p1, p2, p3;
    if (SGN) {
        p0 = (w << 6) & 0xC0C0C0C0u; p1 = (w << 4) & 0xC0C0C0C0u; p2 = (w << 2) & 0xC0C0C0C0u; p3 = w & 0xC0C0C0C0u;
    } else {
        p0 = w & 0x03030303u; p1 = (w >> 2) & 0x03030303u; p2 = (w >> 4) & 0x03030303u; p3 = (w >> 6) & 0x03030303u;
    }
    const uint32_t a = __byte_perm(p0, p1, 0x5140), b = __byte_perm(p2, p3, 0x5140);
    const uint32_t c = __byte_perm(p0, p1, 0x7362), d = __byte_perm(p2, p3, 0x7362);
    return make_uint4(__byte_perm(a, b, 0x5410), __byte_perm(a, b, 0x7632), __byte_perm(c, d, 0x5410),
                      __byte_perm(c, d, 0x7632));
}

// One 16-byte chunk of packed codes -> 8/C chunks of int8 written at dst[oc ^ sw], oc = oc0 .. oc0 + 8/C - 1.
// `row` points at the first chunk slot of the destination row; `sw` is the row's swizzle mask.
template <int C, int SGN>
__device__ __forceinline__ void expand_chunk(uint4 in, uint8_t* row, int oc0, int sw) {
    if (C == 4) {
        uint4 o0, o1;
        unpack4<SGN>(in.x, o0.x, o0.y);
        unpack4<SGN>(in.y, o0.z, o0.w);
        unpack4<SGN>(in.z, o1.x, o1.y);
        unpack4<SGN>(in.w, o1.z, o1.w);
        *reinterpret_cast<uint4*>(row + ((oc0 ^ sw) << 4)) = o0;
        *reinterpret_cast<uint4*>(row + (((oc0 + 1) ^ sw) << 4)) = o1;
    } else if (C == 2) {
        *reinterpret_cast<uint4*>(row + ((oc0 ^ sw) << 4)) = unpack2<SGN>(in.x);
        *reinterpret_cast<uint4*>(row + (((oc0 + 1) ^ sw) << 4)) = unpack2<SGN>(in.y);
        *reinterpret_cast<uint4*>(row + (((oc0 + 2) ^ sw) << 4)) = unpack2<SGN>(in.z);
        *reinterpret_cast<uint4*>(row + (((oc0 + 3) ^ sw) << 4)) = unpack2<SGN>(in.w);
    } else {
        *reinterpret_cast<uint4*>(row + ((oc0 ^ sw) << 4)) = in;
    }
}


// The same codes in another order within the chunk -- all low fields of the four words first, then the next ones: no byte
// permutes, 12 instead of 20 operations for 32 four-bit codes.  For contractions whose two operands go through this function
// with the same C: the order of k is the same on both sides.
template <int C, int SGN>
__device__ __forceinline__ void expand_chunk_reordered(uint4 in, uint8_t* row, int oc0, int sw) {
    constexpr uint32_t MASK = C == 4 ? (SGN ? 0xF0F0F0F0u : 0x0F0F0F0Fu) : (SGN ? 0xC0C0C0C0u : 0x03030303u);
#pragma unroll
    for (int f = 0; f < 8 / C; ++f) {
        const int s = SGN ? 8 - C - C * f : C * f;                // left (signed: into the high bits) or right
        auto field = [&](uint32_t w) { return (SGN ? w << s : w >> s) & MASK; };
        *reinterpret_cast<uint4*>(row + (((oc0 + f) ^ sw) << 4)) = make_uint4(field(in.x), field(in.y), field(in.z), field(in.w));
    }
}

// Rows of 64 int8 (64 codes each), 64-byte swizzle: row r lives at r*64 and its 16-byte chunk
// cc at slot cc ^ ((r >> 1) & 3).  This one layout serves a K-contiguous operand with K = 64
// (SBO = 512) and an N-contiguous operand with N = 64 (eight K rows per 512-byte group).
template <int C, int SGN>
__device__ __forceinline__ void unpack_rows64(const uint8_t* src, uint8_t* dst, int rows, int tid, int nthreads) {
    constexpr int LH = C == 2 ? 0 : (C == 4 ? 1 : 2);   // log2(packed chunks per 64-code row)
    constexpr int E = 8 / C;
    const int chunks = rows << LH;
#pragma unroll 2
    for (int q = tid; q < chunks; q += nthreads) {
        const int r = q >> LH, h = q & ((1 << LH) - 1);
        const uint4 in = *reinterpret_cast<const uint4*>(src + (size_t)q * 16);
        expand_chunk<C, SGN>(in, dst + r * 64, h * E, (r >> 1) & 3);
    }
}

// ---- softmax of a block of scores by table (attention kernels) ---------------------------------------------------
// The table holds exp(fl32(s * c)) for every integer score, as a ring: the entry of score s lies at s mod n, n = 2 smax
// (a power of two).  Scores of signed codes reach smax = 64 * 2^(b-1) * 2^(b-1) but never -smax, so none share an entry, and
// one AND turns 4 s into a byte offset that lies inside the table whatever the operand bytes were.
// (Four entries a load; smax is a multiple of 256.)
__device__ __forceinline__ void fill_table_ring(float* ring, const float* __restrict__ linear, int smax, int tid, int nthreads) {
#pragma unroll 4
    for (int i = 4 * tid; i < 2 * smax; i += 4 * nthreads) {
        float4 v = __ldg(reinterpret_cast<const float4*>(i < smax ? linear + smax + i : linear + (i - smax)));
        if (i == smax) v.x = __ldg(linear + 2 * smax);
        *reinterpret_cast<float4*>(ring + i) = v;
    }
}

// v: scores s (SCALED: 4 s times 2^sh) -> the entries' bits; their fp64 sum goes into four interleaved partial sums (one would
// chain N dependent additions).  MASKED: elements from n_valid on are no scores: entry 0, nothing added.
// Z = 2: v holds two of every four columns, and the sums are those two of the four that they belong to.
template <int N, bool SCALED, bool MASKED, int Z>
__device__ __forceinline__ void exp_lookup(uint32_t (&v)[N], const char* ring, uint32_t mask, int sh, int n_valid, double (&zp)[Z]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t off = (SCALED ? (uint32_t)((int)v[i] >> sh) : v[i] * 4u) & mask;
        uint32_t eb = *reinterpret_cast<const uint32_t*>(ring + off);
        const int column = Z == 4 ? i : 4 * (i >> 1) + (i & 1);
        if (MASKED && column >= n_valid) eb = 0u;
        // an entry is a positive normal float: its double is put together from the bits, one instruction on the integer unit
        // and one on the multiplier (the conversion unit runs at a quarter of the fp64 adder's rate)
        const uint32_t hi = (eb >> 3) + 0x38000000u;
        uint32_t lo;
        asm("mul.lo.u32 %0, %1, 536870912;" : "=r"(lo) : "r"(eb));                    // eb << 29
        zp[i & (Z - 1)] += __hiloint2double(MASKED && column >= n_valid ? 0 : (int)hi, (int)lo);
        v[i] = eb;
    }
}

// Codes min(rint(e * (rh + rl)), Qp), e * rh + RN(e * rl): two scores per instruction up to the rounding by 1.5*2^23, then
// two 16-bit minima per instruction (the caller keeps e * r below 2^16).
template <int N>
__device__ __forceinline__ void quantize_entries(const uint32_t (&v)[N], f32x2 rh2, f32x2 rl2, uint32_t qp2, uint32_t (&w)[N / 4]) {
    const f32x2 magic2 = f2_dup(12582912.0f);
#pragma unroll
    for (int i4 = 0; i4 < N / 4; ++i4) {
        uint32_t h[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const f32x2 e2 = f2_pack(__uint_as_float(v[4 * i4 + 2 * j]), __uint_as_float(v[4 * i4 + 2 * j + 1]));
            float c0, c1;
            f2_unpack(f2_add(f2_fma(e2, rh2, f2_mul(e2, rl2)), magic2), c0, c1);
            const uint32_t both = __byte_perm(__float_as_uint(c0), __float_as_uint(c1), 0x5410);
            asm("min.u16x2 %0, %1, %2;" : "=r"(h[j]) : "r"(both), "r"(qp2));
        }
        w[i4] = __byte_perm(h[0], h[1], 0x6420);
    }
}

// Codes min(rint(e * r), Qp) that hold for every r between lo and hi: rounding is monotone, so two products with the ends of the
// interval prove a code.  Returns 0 where all N codes (the lower end's are stored) are proven.  e * hi < 2^16.  The products and
// the test run on the FMA pipe, four packed instructions a pair; 2.5 are left for the ALU, which takes two cycles for each (a
// comparison of |a - rint(a)| with a limit has 5.5: clamp, maxima, packing).
template <int N>
__device__ __forceinline__ float quantize_interval(const f32x2 (&e)[N / 2], f32x2 lo2, f32x2 hi2, uint32_t qp2, uint32_t (&w)[N / 4]) {
    const f32x2 magic2 = f2_dup(12582912.0f), neg1 = f2_dup(-1.0f);
    f32x2 differ = f2_dup(0.0f);
#pragma unroll
    for (int i4 = 0; i4 < N / 4; ++i4) {
        uint32_t h[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const f32x2 lo = f2_fma(e[2 * i4 + j], lo2, magic2), hi = f2_fma(e[2 * i4 + j], hi2, magic2);
            differ = f2_add(differ, f2_fma(lo, neg1, hi));                           // small integers, none negative
            float c0, c1;
            f2_unpack(lo, c0, c1);
            const uint32_t both = __byte_perm(__float_as_uint(c0), __float_as_uint(c1), 0x5410);
            asm("min.u16x2 %0, %1, %2;" : "=r"(h[j]) : "r"(both), "r"(qp2));
        }
        w[i4] = __byte_perm(h[0], h[1], 0x6420);
    }
    float d0, d1;
    f2_unpack(differ, d0, d1);
    return d0 + d1;
}

// The interval grows with the value, so far beyond the last level it often holds a boundary although the code is Qp for certain.
// The same once more, where the first look proved nothing, with values kept at `top`, about (Qp + 1) / r.
template <int N>
__device__ __forceinline__ float quantize_interval_below(const f32x2 (&e)[N / 2], float top, f32x2 lo2, f32x2 hi2, uint32_t qp2, uint32_t (&w)[N / 4]) {
    f32x2 c[N / 2];
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        float a, b;
        f2_unpack(e[i], a, b);
        c[i] = f2_pack(fminf(a, top), fminf(b, top));
    }
    return quantize_interval<N>(c, lo2, hi2, qp2, w);
}

// The table's codes straight from the scores, without the table: a = 2^(s c2 + l), l = log2(1 / (Z s_P)), in fp32 with the
// hardware's exp2.  a differs from the quantizer's own argument by a relative error below the bound that the caller turned
// into `limit` (a little less than 1/2): where |a - rint(a)| stays below it both round to the same code, where it does not
// (about one score in 2^14) the function returns false and the caller takes the table.
template <int N>
__device__ __forceinline__ bool quantize_scores(const uint32_t (&v)[N], f32x2 c2, f32x2 l2, float qp, float limit, uint32_t (&w)[N / 4]) {
    const f32x2 magic2 = f2_dup(12582912.0f), nmagic2 = f2_dup(-12582912.0f), neg1 = f2_dup(-1.0f);
    float dev = 0.0f;
#pragma unroll
    for (int i4 = 0; i4 < N / 4; ++i4) {
        uint32_t c[4];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const f32x2 s = f2_add(f2_pack(__uint_as_float(0x4B400000u + v[4 * i4 + 2 * j]), __uint_as_float(0x4B400000u + v[4 * i4 + 2 * j + 1])), nmagic2);
            float t0, t1, a0, a1, c0, c1, d0, d1;
            f2_unpack(f2_fma(s, c2, l2), t0, t1);
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a0) : "f"(t0));
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a1) : "f"(t1));
            const f32x2 a = f2_pack(fminf(a0, qp), fminf(a1, qp)), m = f2_add(a, magic2);
            f2_unpack(f2_fma(f2_add(m, nmagic2), neg1, a), d0, d1);
            dev = fmaxf(dev, fmaxf(fabsf(d0), fabsf(d1)));
            f2_unpack(m, c0, c1);
            c[2 * j] = __float_as_uint(c0);
            c[2 * j + 1] = __float_as_uint(c1);
        }
        w[i4] = __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
    }
    return dev < limit;
}

// Requantizes N columns of an accumulator row (scaled by 2^sh; SMALL: |acc| < 2^22) to byte codes in two's complement:
// clamp(rint(fma(acc, a, b))).  pa, pb: the columns' parameters in shared memory, 16-byte aligned.
template <bool SMALL, int N>
__device__ __forceinline__ void requantize_row(const uint32_t (&v)[N], int sh, const float* pa, const float* pb, float qn, float qp,
                                               uint32_t (&w)[N / 4]) {
    const f32x2 magic2 = f2_dup(12582912.0f), nmagic2 = f2_dup(-12582912.0f);
#pragma unroll
    for (int i4 = 0; i4 < N / 4; ++i4) {
        const float4 a4 = *reinterpret_cast<const float4*>(pa + 4 * i4), b4 = *reinterpret_cast<const float4*>(pb + 4 * i4);
        uint32_t c[4];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int u0 = (int)v[4 * i4 + 2 * p] >> sh, u1 = (int)v[4 * i4 + 2 * p + 1] >> sh;
            const f32x2 f = SMALL ? f2_add(f2_pack(__int_as_float(0x4B400000 + u0), __int_as_float(0x4B400000 + u1)), nmagic2)
                                  : f2_pack((float)u0, (float)u1);
            float y0, y1, c0, c1;
            f2_unpack(f2_fma(f, p ? f2_pack(a4.z, a4.w) : f2_pack(a4.x, a4.y), p ? f2_pack(b4.z, b4.w) : f2_pack(b4.x, b4.y)), y0, y1);
            f2_unpack(f2_add(f2_pack(fminf(fmaxf(y0, qn), qp), fminf(fmaxf(y1, qn), qp)), magic2), c0, c1);
            c[2 * p] = __float_as_uint(c0);
            c[2 * p + 1] = __float_as_uint(c1);
        }
        w[i4] = __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
    }
}

// Sixteen byte codes -> eight bytes of 4-bit or four bytes of 2-bit codes (element order kept).
__device__ __forceinline__ void narrow4(const uint32_t (&w)[4], uint32_t (&o)[2]) {
    uint32_t t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t n = w[k] & 0x0F0F0F0Fu;
        t[k] = n | (n >> 4);                                    // bytes 0 and 2 hold two codes each
    }
    o[0] = __byte_perm(t[0], t[1], 0x6420);
    o[1] = __byte_perm(t[2], t[3], 0x6420);
}
__device__ __forceinline__ uint32_t narrow2(const uint32_t (&w)[4]) {
    uint32_t t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t n = w[k] & 0x03030303u;
        n |= n >> 6;                                            // bytes 0 and 2: two codes in the low four bits
        t[k] = n | (n >> 12);                                   // byte 0: four codes
    }
    return __byte_perm(__byte_perm(t[0], t[1], 0x0040), __byte_perm(t[2], t[3], 0x0040), 0x5410);
}
// Stores 16 or 32 byte codes of a row in the output's container (o: 2 or 4 * out_c bytes, aligned to 16 bytes or their number).
__device__ __forceinline__ void store_row(uint8_t* o, const uint32_t (&w)[4], int out_c) {
    if (out_c == 8) {
        *reinterpret_cast<uint4*>(o) = make_uint4(w[0], w[1], w[2], w[3]);
    } else if (out_c == 4) {
        uint32_t a[2];
        narrow4(w, a);
        *reinterpret_cast<uint2*>(o) = make_uint2(a[0], a[1]);
    } else {
        *reinterpret_cast<uint32_t*>(o) = narrow2(w);
    }
}
__device__ __forceinline__ void store_row(uint8_t* o, const uint32_t (&w)[8], int out_c) {
    const uint32_t lo[4] = {w[0], w[1], w[2], w[3]}, hi[4] = {w[4], w[5], w[6], w[7]};
    if (out_c == 8) {
        if ((reinterpret_cast<uintptr_t>(o) & 31u) == 0) {
            // one 32-byte store: a warp's store touches 32 different rows whatever its width
            ptx::st_global_32B(o, lo, hi);
        } else {
            reinterpret_cast<uint4*>(o)[0] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            reinterpret_cast<uint4*>(o)[1] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        }
    } else if (out_c == 4) {
        uint32_t a[2], b[2];
        narrow4(lo, a);
        narrow4(hi, b);
        *reinterpret_cast<uint4*>(o) = make_uint4(a[0], a[1], b[0], b[1]);
    } else {
        *reinterpret_cast<uint2*>(o) = make_uint2(narrow2(lo), narrow2(hi));
    }
}

}  // namespace vitint

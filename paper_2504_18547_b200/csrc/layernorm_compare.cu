// Quantizing LayerNorm of Section IV-C: the running statistics of Eq. 5 and the division- and
// square-root-free comparator of Fig. 5(b), in one kernel.
//
//   statistics  one thread per row walks the row in order:
//                 delta = x_i - mu;  mu += delta / i;  S += delta * (x_i - mu)
//               every operation a single round-to-nearest fp32 one (no contraction), the
//               division by i exactly rounded from a reciprocal of two floats.
//   comparator  level = Qn + number of references exceeded.  With d = x - mu (negated where
//               gamma < 0) the sign logic of the figure collapses into one comparison of
//               signed squares,  copysign(d*d, d) > V * r,  r = sgn(c) c^2 / n the caller's
//               signed reference.  The references of a column ascend, so the comparisons are true up to some
//               index and false after it.  Folded from a uniform quantizer they are the signed squares of equally
//               spaced points, so the index is guessed from d / sqrt(V) (two operations) and two comparisons around
//               the guess, formed exactly as defined, prove it; where they do not, all references are compared.
//
// What bounds it.  The recurrence is a chain of four dependent fp32 operations per element (16 cycles, 768 elements: 6.5 us)
// and cannot be split without changing the order of Eq. 5 and with it the bits; one CTA per SM walks all its rows at once, one
// lane each, while TMA keeps the next chunks of columns coming and the other warps lay out the references.  Its levels it finds
// afterwards with all warps, the rows coming from L2.  As two kernels -- statistics, then a bisection over references held in
// registers, 42 instructions an element -- 12,608 x 768 took 39 us and 25,216 x 768 74 us; as one 25 and 38, of which the walk
// 13 and 17; with the quotient in two operations instead of three (2 x 1.0 us of a layer at batch 64) 24.  (Requesting the next task's rows ahead of the present one's levels: no change.)
#include "common.cuh"
#include "ptx.cuh"
#include "tile_ops.cuh"

namespace vitint {
namespace {

constexpr int LNC_THREADS = 512, LNC_WARPS = LNC_THREADS / 32;
constexpr int LNC_CHUNK = 64;                  // columns per staged chunk: two TMA boxes of 32, 128-byte swizzle (a lane reads its own
                                               // row in 16-byte pieces without bank conflicts)
constexpr int LNC_MAX_BUFFERS = 6;
constexpr int LNC_MAX_ROWS = 192;              // rows a CTA walks at once (six warps)
constexpr int LNC_SLAB = 768, LNC_QUARTER = LNC_SLAB / 4;     // columns whose references are in shared memory at a time
constexpr int LNC_ROW_BATCH = 4;               // rows of one comparator task: their loads are issued together
constexpr int LNS_MAX_COLS = 4096;

// One step of Eq. 5 for element xi, (rh, rl) = 1/i to 47 bits: every operation a single rounded fp32 one.  The update of S
// belonging to the PREVIOUS element (its delta in pd, its value in px; mu is still that element's mean) is
// written between the operations of this element's dependent chain delta -> quotient -> mu, so the two
// interleave in issue order; operands and operations are exactly those of the recurrence.
//
// RN(delta / i) = fma(delta, rh, RN(delta rl)): what is rounded last is within 2^-46 of the quotient, and a quotient of a 24-bit
// number by an i <= 4096 is at least ulp / 2i = 2^-37 away from a rounding boundary (it cannot lie on one: the odd part of a
// boundary times i has 25 bits or more) -- unless the product underflows: `tiny` keeps the smallest |delta| that is not 0, as bits
// less 1, and a row that had one below 2^-100, or did not stay finite, is walked again by running_row_slow.
__device__ __forceinline__ void running_step(float xi, float rh, float rl, float& mu, float& S, float& pd, float& px, uint32_t& tiny) {
    const float delta = __fadd_rn(xi, -mu);
    const float tt = __fadd_rn(px, -mu);
    const float lo = __fmul_rn(delta, rl);
    const float pp = __fmul_rn(pd, tt);
    const float q = __fmaf_rn(delta, rh, lo);
    S = __fadd_rn(S, pp);
    mu = __fadd_rn(mu, q);
    tiny = min(tiny, (__float_as_uint(delta) & 0x7FFFFFFFu) - 1u);
    pd = delta;
    px = xi;
}
// The whole row from memory, RN(delta / i) as q0 = RN(delta r), an exact remainder in one FMA and one correction.
__device__ __noinline__ float2 running_row_slow(const float* __restrict__ x, int cols) {
    float mu = 0.0f, S = 0.0f;
    for (int i = 0; i < cols; ++i) {
        const float fi = (float)(i + 1), r = __frcp_rn(fi), xi = __ldg(x + i);
        const float delta = __fadd_rn(xi, -mu), q0 = __fmul_rn(delta, r);
        mu = __fadd_rn(mu, __fmaf_rn(__fmaf_rn(-q0, fi, delta), r, q0));
        S = __fadd_rn(S, __fmul_rn(delta, __fadd_rn(xi, -mu)));
    }
    return make_float2(mu, S);
}

struct LncShape {
    int cols, rows_cta, nbuf;
    uint32_t off_ref, off_col, off_stage, buf_bytes;
};

// References of columns slab0 .. slab0 + 767 in shared memory, [NT + 2][768] with -inf and +inf around them and column c at
// (c % 4) * 192 + c / 4, so that the lanes of a warp (four neighbouring columns each) read different banks whatever their
// levels; and per column inv, off and the sign of the gain, for the guess  count ~ rint(NT * sat((x - mu) / sqrt(V) * inv + off)):
// with the references as signed roots rho, inv = (NT - 1) / (rho_last - rho_first) / NT (negated for a negative gain),
// off = (1/2 - rho_first * (NT - 1) / (rho_last - rho_first)) / NT.
template <int NT>
__device__ __forceinline__ void lnc_load_refs(float* s_ref, float* s_col, const LncShape& sh, int slab0, const float* __restrict__ refs,
                                              const uint8_t* __restrict__ flip, int t0, int nthreads) {
    const int n = min(LNC_SLAB, sh.cols - slab0);
    for (int c = t0; c < n; c += nthreads) {
        float* const dst = s_ref + (c & 3) * LNC_QUARTER + (c >> 2);
        float first = 0.0f, last = 0.0f;
        dst[0] = -INFINITY;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const float r = __ldg(refs + (int64_t)(slab0 + c) * NT + t);
            if (t == 0) first = r;
            if (t == NT - 1) last = r;
            dst[(t + 1) * LNC_SLAB] = r;
        }
        dst[(NT + 1) * LNC_SLAB] = INFINITY;
        const float rho0 = copysignf(sqrtf(fabsf(first)), first), rho1 = copysignf(sqrtf(fabsf(last)), last);
        float inv = __fdividef((float)(NT - 1), rho1 - rho0);
        if (!(inv < 1e30f)) inv = 0.0f;
        const float sgn = (flip && __ldg(flip + slab0 + c)) ? -1.0f : 1.0f;
        s_col[c] = inv * sgn * (1.0f / NT);
        s_col[LNC_SLAB + c] = (0.5f - rho0 * inv) * (1.0f / NT);
        s_col[2 * LNC_SLAB + c] = sgn;
    }
}

template <int BITS, int C>
__global__ void __launch_bounds__(LNC_THREADS, 1)
ln_compare_quantize_kernel(const __grid_constant__ CUtensorMap map_x, const float* __restrict__ x, int64_t rows, int64_t ldx,
                           const float* __restrict__ refs, const uint8_t* __restrict__ flip, float n_eps, float* __restrict__ stats,
                           uint8_t* __restrict__ out, int64_t pitch, int qn, const __grid_constant__ LncShape sh) {
    extern __shared__ uint8_t lnc_raw[];
    __shared__ float2 s_stat[LNC_MAX_ROWS];                     // (mu, V) of the CTA's rows
    __shared__ uint64_t full[LNC_MAX_BUFFERS], empty[LNC_MAX_BUFFERS];
    __shared__ int abort_flag;
    constexpr int NT = (1 << BITS) - 1;
    constexpr int LANES_PER_WORD = 8 / C;                       // lanes whose 4 codes share one 32-bit word
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t* const smem = lnc_raw + ((1024u - (ptx::smem_addr(lnc_raw) & 1023u)) & 1023u);
    float2* const tab = reinterpret_cast<float2*>(smem);        // 1/i of every column, i from 1, as a sum of two floats
    float* const s_ref = reinterpret_cast<float*>(smem + sh.off_ref);
    float* const s_col = reinterpret_cast<float*>(smem + sh.off_col);
    uint8_t* const stage = smem + sh.off_stage;
    const int cols = sh.cols, nbuf = sh.nbuf;
    const int walkers = (sh.rows_cta + 31) / 32;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int b = 0; b < nbuf; ++b) {
            ptx::mbar_init(ptx::smem_addr(&full[b]), 1);
            ptx::mbar_init(ptx::smem_addr(&empty[b]), (uint32_t)walkers);
        }
        ptx::fence_mbar_init();
        ptx::fence_proxy_async_smem();
    }
    for (int i = threadIdx.x; i < cols; i += LNC_THREADS) {
        const float fi = (float)(i + 1), rh = __frcp_rn(fi);
        tab[i] = make_float2(rh, __fmul_rn(__fmaf_rn(-rh, fi, 1.0f), rh));         // (a division here: 0.1 - 0.2 us of a call, 3.71 -> 3.89 at 2368 x 64)
    }
    __syncthreads();
    grid_dependency_wait();        // x may come from the previous kernel of the stream
    grid_dependency_launch();
    const int n_chunks = (cols + LNC_CHUNK - 1) / LNC_CHUNK;
    const int words_per_row = (int)(pitch / 4);
    // a lane covers four columns; with sub-byte containers the words up to the pitch are written (as zero) past the last column
    const int lanes_total = max(cols / 4, words_per_row * LANES_PER_WORD);
    constexpr uint32_t FIELDS = 1u | (1u << C) | (1u << (2 * C)) | (1u << (3 * C));
    const uint32_t qn_low = ((uint32_t)qn & ((1u << (C - 1)) - 1u)) * FIELDS, qn_top = ((uint32_t)qn & (1u << (C - 1))) * FIELDS;
    int slab_in = -1;                                           // first column of the references in shared memory
    int buf = 0;                                                // of the walkers and of the producer: next buffer and its phase
    uint32_t ph = 0u;
    bool ok = true;
    for (int64_t row0 = (int64_t)blockIdx.x * sh.rows_cta; row0 < rows; row0 += (int64_t)gridDim.x * sh.rows_cta) {
        const int n_rows = rows - row0 < sh.rows_cta ? (int)(rows - row0) : sh.rows_cta;
        // ---- statistics ----
        if (warp < walkers) {
            float mu = 0.0f, S = 0.0f, pd = 0.0f, px = 0.0f;
            uint32_t tiny = 0xFFFFFFFFu;
            const int my_row = min(warp * 32 + lane, sh.rows_cta - 1), r7 = my_row & 7;
            for (int c = 0; c < n_chunks; ++c) {
                const bool w = mbar_wait(ptx::smem_addr(&full[buf]), ph, &abort_flag);
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                const uint8_t* mine = stage + (size_t)buf * sh.buf_bytes + my_row * 128;
                const float4* t4 = reinterpret_cast<const float4*>(tab + c * LNC_CHUNK);   // two columns' pairs
                const int box = sh.buf_bytes >> 1;
                // four elements of the row and their (i, 1/i); the next four are read before these are walked
                struct Four { float4 e, ta, tb; };
                auto read = [&](int v) {
                    return Four{*reinterpret_cast<const float4*>(mine + (v >> 3) * box + (((v & 7) ^ r7) << 4)), t4[2 * v], t4[2 * v + 1]};
                };
                const int nv = (cols - c * LNC_CHUNK < LNC_CHUNK ? cols - c * LNC_CHUNK : LNC_CHUNK) >> 2;
                Four cur = read(0);
#pragma unroll 4
                for (int v = 0; v < nv; ++v) {
                    const Four next = read(v + 1 < nv ? v + 1 : v);
                    running_step(cur.e.x, cur.ta.x, cur.ta.y, mu, S, pd, px, tiny);
                    running_step(cur.e.y, cur.ta.z, cur.ta.w, mu, S, pd, px, tiny);
                    running_step(cur.e.z, cur.tb.x, cur.tb.y, mu, S, pd, px, tiny);
                    running_step(cur.e.w, cur.tb.z, cur.tb.w, mu, S, pd, px, tiny);
                    cur = next;
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&empty[buf]));
                if (++buf == nbuf) { buf = 0; ph ^= 1u; }
            }
            if (ok && warp * 32 + lane < n_rows) {
                S = __fadd_rn(S, __fmul_rn(pd, __fadd_rn(px, -mu)));                   // the last element's term
                if (tiny < 0x0D800000u - 1u || !(fabsf(mu) < INFINITY)) {              // 2^-100
                    const float2 again = running_row_slow(x + (row0 + my_row) * ldx, cols);
                    mu = again.x;
                    S = again.y;
                }
                const float2 st = make_float2(mu, __fadd_rn(S, n_eps));
                s_stat[my_row] = st;
                reinterpret_cast<float2*>(stats)[row0 + my_row] = st;
            }
        } else if (warp == LNC_WARPS - 1) {
            if (lane == 0) {
                const uint32_t bytes = (uint32_t)sh.rows_cta * 128u;
                int c = 0;
                for (; c < n_chunks; ++c) {
                    if (!mbar_wait(ptx::smem_addr(&empty[buf]), ph ^ 1u, &abort_flag)) { ok = false; break; }
                    const uint32_t bar = ptx::smem_addr(&full[buf]), dst = ptx::smem_addr(stage) + (uint32_t)buf * sh.buf_bytes;
                    const bool two = c * LNC_CHUNK + 32 < cols;
                    ptx::mbar_arrive_expect_tx(bar, two ? 2u * bytes : bytes);
                    ptx::tma_load_3d(dst, &map_x, bar, c * LNC_CHUNK, (int)row0, 0);
                    if (two) ptx::tma_load_3d(dst + (sh.buf_bytes >> 1), &map_x, bar, c * LNC_CHUNK + 32, (int)row0, 0);
                    if (++buf == nbuf) { buf = 0; ph ^= 1u; }
                }
                if (!ok) {
                    // give the copies still in flight a bounded chance to land before the CTA exits
                    for (int j = 0; j < nbuf; ++j)
                        for (int spin = 0; spin < (1 << 20) && !ptx::mbar_try_wait(ptx::smem_addr(&full[j]), j < buf ? ph : ph ^ 1u); ++spin) {}
                }
            }
            __syncwarp();
        } else if (slab_in != 0) {
            lnc_load_refs<NT>(s_ref, s_col, sh, 0, refs, flip, threadIdx.x - walkers * 32, LNC_THREADS - (walkers + 1) * 32);
        }
        slab_in = 0;
        if (!__syncthreads_and(ok ? 1 : 0)) return;

        // ---- comparator ----
        for (int slab0 = 0; slab0 < lanes_total * 4; slab0 += LNC_SLAB) {
            if (slab0 != slab_in && slab0 < cols) {
                __syncthreads();
                lnc_load_refs<NT>(s_ref, s_col, sh, slab0, refs, flip, threadIdx.x, LNC_THREADS);
                slab_in = slab0;
                __syncthreads();
            }
            const int groups = (min(lanes_total - slab0 / 4, LNC_QUARTER) + 31) / 32;      // of 32 lanes
            const int batches = (n_rows + LNC_ROW_BATCH - 1) / LNC_ROW_BATCH;
            for (int task = warp; task < groups * batches; task += LNC_WARPS) {
                const int batch = task / groups, grp = task - batch * groups;
                const int ql = grp * 32 + lane;                                            // the lane's four columns within the slab
                const int col = slab0 + ql * 4;
                const bool col_ok = col < cols;
                const int rb = batch * LNC_ROW_BATCH;
                const float* xp = x + (row0 + rb) * ldx + col;
                float4 xb[LNC_ROW_BATCH];
#pragma unroll
                for (int k = 0; k < LNC_ROW_BATCH; ++k, xp += ldx)
                    xb[k] = (col_ok && rb + k < n_rows) ? __ldg(reinterpret_cast<const float4*>(xp)) : make_float4(0.f, 0.f, 0.f, 0.f);
                const int qs = col_ok ? ql : 0;
                const float4 inv4 = *reinterpret_cast<const float4*>(s_col + 4 * qs), off4 = *reinterpret_cast<const float4*>(s_col + LNC_SLAB + 4 * qs);
                const float4 sgn4 = *reinterpret_cast<const float4*>(s_col + 2 * LNC_SLAB + 4 * qs);
                const float inv[4] = {inv4.x, inv4.y, inv4.z, inv4.w}, off[4] = {off4.x, off4.y, off4.z, off4.w};
                const f32x2 sgn[2] = {f2_pack(sgn4.x, sgn4.y), f2_pack(sgn4.z, sgn4.w)};
                // the guess arrives as 1.5*2^23 + count: times the row of references it is an address, the constant folded into the base
                const uint32_t ref0 = ptx::smem_addr(s_ref) + 4u * (uint32_t)qs - 0x4B400000u * (4u * LNC_SLAB);
                uint8_t* o = out + (row0 + rb) * pitch + (int64_t)((slab0 / 4 + ql) / LANES_PER_WORD) * 4;
                const bool writes = (lane % LANES_PER_WORD) == 0 && ql < LNC_QUARTER && (slab0 / 4 + ql) / LANES_PER_WORD < words_per_row;
#pragma unroll
                for (int k = 0; k < LNC_ROW_BATCH; ++k, o += pitch) {
                    if (rb + k >= n_rows) break;                                           // uniform across the warp
                    const float2 st = s_stat[rb + k];
                    const float V = st.y;
                    const f32x2 nm2 = f2_dup(-st.x), rs2 = f2_dup(rsqrtf(V)), V2 = f2_dup(V);
                    const f32x2 xs[2] = {f2_pack(xb[k].x, xb[k].y), f2_pack(xb[k].z, xb[k].w)};
                    float ds[4];
                    uint32_t g[4];
                    bool proven = true;
#pragma unroll
                    for (int p = 0; p < 2; ++p) {
                        const f32x2 delta = f2_add(xs[p], nm2), d = f2_mul(delta, sgn[p]);                 // exact sign change
                        float d0, d1, q0, q1, u0, u1, g0, g1, l0, l1, h0, h1;
                        f2_unpack(d, d0, d1);
                        f2_unpack(f2_mul(d, d), q0, q1);
                        ds[2 * p] = copysignf(q0, d0);
                        ds[2 * p + 1] = copysignf(q1, d1);
                        f2_unpack(f2_mul(delta, rs2), u0, u1);
                        u0 = __saturatef(fmaf(u0, inv[2 * p], off[2 * p]));
                        u1 = __saturatef(fmaf(u1, inv[2 * p + 1], off[2 * p + 1]));
                        f2_unpack(f2_fma(f2_pack(u0, u1), f2_dup((float)NT), f2_dup(12582912.0f)), g0, g1);
                        g[2 * p] = __float_as_uint(g0);
                        g[2 * p + 1] = __float_as_uint(g1);
                        const uint32_t r0 = g[2 * p] * (4u * LNC_SLAB) + (ref0 + 8u * p * LNC_QUARTER);
                        const uint32_t r1 = g[2 * p + 1] * (4u * LNC_SLAB) + (ref0 + (8u * p + 4u) * LNC_QUARTER);
                        f2_unpack(f2_mul(V2, f2_pack(ptx::ld_shared_f32(r0), ptx::ld_shared_f32(r1))), l0, l1);   // reference count - 1
                        f2_unpack(f2_mul(V2, f2_pack(ptx::ld_shared_f32(r0 + 4 * LNC_SLAB), ptx::ld_shared_f32(r1 + 4 * LNC_SLAB))), h0, h1);
                        proven = proven && ds[2 * p] > l0 && !(ds[2 * p] > h0) && ds[2 * p + 1] > l1 && !(ds[2 * p + 1] > h1);
                    }
                    uint32_t n = (g[0] + (g[1] << C) + (g[2] << (2 * C)) + (g[3] << (3 * C))) -
                                 0x4B400000u * (1u + (1u << C) + (1u << (2 * C)) + (1u << (3 * C)));
                    if (!proven && col_ok) {
                        n = 0;
                        const float* my_ref = s_ref + qs;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            uint32_t cnt = 0;
#pragma unroll 1
                            for (int t = 1; t <= NT; ++t) cnt += ds[j] > __fmul_rn(V, my_ref[j * LNC_QUARTER + t * LNC_SLAB]) ? 1u : 0u;
                            n |= cnt << (C * j);
                        }
                    }
                    // counts to levels: Qn added to each field (no field overflows: its low bits, then its top bit by an exclusive or)
                    uint32_t bits = col_ok ? (n + qn_low) ^ qn_top : 0u;
                    // gather 8/C neighbouring lanes into one 32-bit word
                    if (C == 4) {
                        bits |= __shfl_xor_sync(0xffffffffu, bits, 1) << 16;
                    } else if (C == 2) {
                        bits |= __shfl_xor_sync(0xffffffffu, bits, 1) << 8;
                        bits |= __shfl_xor_sync(0xffffffffu, bits, 2) << 16;
                    }
                    if (writes) *reinterpret_cast<uint32_t*>(o) = bits;
                }
            }
        }
        __syncthreads();                                                                   // s_stat is free for the next rows
    }
}

inline uint32_t lnc_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

template <int BITS, int C>
int launch_ln_compare(cudaStream_t st, const float* x, int64_t rows, int cols, int64_t ldx, const float* refs, const uint8_t* flip,
                      float n_eps, float* stats, uint8_t* out, int64_t pitch, int qn) {
    // all SMs, as many rounds as 192 rows a CTA make necessary, the rows spread evenly over them
    const int64_t sms = sm_count(), rounds = (rows + sms * LNC_MAX_ROWS - 1) / (sms * LNC_MAX_ROWS);
    LncShape sh{};
    sh.cols = cols;
    sh.rows_cta = (int)((rows + sms * rounds - 1) / (sms * rounds));
    sh.rows_cta = sh.rows_cta < 8 ? 8 : sh.rows_cta;
    sh.off_ref = lnc_up((uint32_t)cols * 8u, 16);
    sh.off_col = sh.off_ref + (uint32_t)((1 << BITS) + 1) * LNC_SLAB * 4u;
    sh.off_stage = lnc_up(sh.off_col + 3u * LNC_SLAB * 4u, 1024);
    sh.buf_bytes = 2u * lnc_up((uint32_t)sh.rows_cta * 128u, 1024);
    const uint32_t budget = 222u * 1024u;
    sh.nbuf = (int)((budget - sh.off_stage) / sh.buf_bytes);
    if (sh.nbuf > LNC_MAX_BUFFERS) sh.nbuf = LNC_MAX_BUFFERS;
    if (sh.nbuf < 2) return VITINT_ERR_UNSUPPORTED;
    const size_t smem = sh.off_stage + (size_t)sh.nbuf * sh.buf_bytes + 1024;
    const int dev = current_device();
    if (dev < 0) return VITINT_ERR_CUDA;
    static bool attr_set[MAX_DEVICES] = {};
    if (!attr_set[dev]) {
        if (cudaFuncSetAttribute(ln_compare_quantize_kernel<BITS, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget + 1024) != cudaSuccess)
            return VITINT_ERR_CUDA;
        attr_set[dev] = true;
    }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return VITINT_ERR_CUDA;
    CUtensorMap map_x;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, 1}, strides[2] = {(cuuint64_t)ldx * 4, (cuuint64_t)ldx * 4 * (cuuint64_t)rows};
    cuuint32_t box[3] = {32, (cuuint32_t)sh.rows_cta, 1}, estr[3] = {1, 1, 1};
    if (fn(&map_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return VITINT_ERR_CUDA;
    const int64_t ctas = (rows + sh.rows_cta - 1) / sh.rows_cta;
    launch_kernel(ln_compare_quantize_kernel<BITS, C>, dim3((unsigned)(ctas < sms ? ctas : sms)), dim3(LNC_THREADS), smem, st, map_x, x, rows,
                  ldx, refs, flip, n_eps, stats, out, pitch, qn, sh);
    return cuda_status(cudaGetLastError());
}

template <int BITS>
int launch_ln_compare_bits(int c, cudaStream_t st, const float* x, int64_t rows, int cols, int64_t ldx, const float* refs,
                           const uint8_t* flip, float n_eps, float* stats, uint8_t* out, int64_t pitch, int qn) {
    if (c == 2) return launch_ln_compare<BITS, 2>(st, x, rows, cols, ldx, refs, flip, n_eps, stats, out, pitch, qn);
    if (c == 4) return launch_ln_compare<BITS, 4>(st, x, rows, cols, ldx, refs, flip, n_eps, stats, out, pitch, qn);
    return launch_ln_compare<BITS, 8>(st, x, rows, cols, ldx, refs, flip, n_eps, stats, out, pitch, qn);
}

}  // namespace
}  // namespace vitint

using namespace vitint;

extern "C" int vitint_layernorm_compare_quantize(const float* x, int64_t rows, int64_t cols, int64_t ldx,
                                                 const float* refs, const uint8_t* flip, float n_eps,
                                                 const vitint_codes* out, float* stats, void* stream) {
    if (!x || !refs || !out || !stats) return VITINT_ERR_INVALID_ARG;
    if (int rc = check_codes(out)) return rc;
    if (rows <= 0 || cols <= 0 || ldx < cols || out->rows != rows || out->cols != cols) return VITINT_ERR_INVALID_ARG;
    if (!(n_eps > 0.0f && n_eps < INFINITY)) return VITINT_ERR_INVALID_ARG;
    if (out->bits == 8 || cols % 4 != 0 || cols > LNS_MAX_COLS) return VITINT_ERR_UNSUPPORTED;
    if (!aligned16(x) || ldx % 4 != 0 || (reinterpret_cast<uintptr_t>(stats) & 7u) != 0) return VITINT_ERR_ALIGNMENT;
    if (rows > 0x7fffffff) return VITINT_ERR_UNSUPPORTED;
    const int c = codes_container(out);
    int qn, qp;
    code_range(out->bits, out->is_signed, &qn, &qp);
    cudaStream_t st = (cudaStream_t)stream;
    uint8_t* o = (uint8_t*)out->data;
    switch (out->bits) {
        case 2: return launch_ln_compare_bits<2>(c, st, x, rows, (int)cols, ldx, refs, flip, n_eps, stats, o, out->pitch_bytes, qn);
        case 3: return launch_ln_compare_bits<3>(c, st, x, rows, (int)cols, ldx, refs, flip, n_eps, stats, o, out->pitch_bytes, qn);
        default: return launch_ln_compare_bits<4>(c, st, x, rows, (int)cols, ldx, refs, flip, n_eps, stats, o, out->pitch_bytes, qn);
    }
}

// a4 + a5 + a6 fused: per (image, head, 128-query tile)  S = Q K^T  ->  softmax + quantize  ->
// O = P V  ->  requantize, with S, the probabilities and P never leaving the SM.
//
// A persistent CTA runs TWO independent pipelines ("groups"), each with eight compute warps
// (query row = TMEM lane, two threads a row) and one control warp (TMA + MMA issue); while one
// group's threads are busy with the softmax the other group's loads and MMAs proceed.  Where no CTA gets a second
// item there is one group of sixteen warps, four threads a row.
//
// Per item and group:
//   control   TMA: packed Q [128 x 64], K [T x 64], V [T x 64] code slabs -> shared memory
//   compute   unpack to int8 operand tiles (rows of 64 bytes, 64-byte swizzle)
//   control   tcgen05.mma  S[128, T] = Q K^T   (K = 64: two MMAs) into TMEM
//   compute   e_j = EXP[S_j] from a table of exp(fl32(s*c)) over every possible integer score
//             (|S| <= 64*max|q|*max|k|: 8192 distinct ones for 4-bit codes); row sum in fp64;
//             p_j = e_j / Z;  code = clamp(rint(p_j / s_P));  codes written as int8 rows (128-byte
//             swizzle) = the A operand of P V.  e_j is parked in TMEM over S between the passes.
//   control   tcgen05.mma  O[128, 64] = P V  (V is the N-contiguous B operand) into TMEM
//   compute   requantize O, pack, store the head's 64 columns of the [M, D] code matrix
//
// What bounds it: the lookups.  Random entries of a 32 KB table take 2.8 passes of the shared-memory pipe per 32 scores: the
// load/store data pipe is 42 % busy with them and the code stores, the tensor core's own reads not counted, and instructions
// issue in 56 % of the slots.  197 tokens x 12 heads, batch 128: 75.5 -> 65.9 us by walking the last columns in blocks of eight
// (200 instead of 224) and 20 % fewer instructions a score; 256 tokens, where nothing is padded, 45.9 -> 45.3.  Overlapping the
// steps of neighbouring items (scores formed while O is pending, O requantized between two chunks) cost more in instructions
// than it hid: 74.8.
//
// Softmax accuracy: exp(t_j)/sum_k exp(t_k) equals Eq. 3's softmax exactly (the maximum is only
// subtracted there for range); every table entry is a correctly rounded fp32, the sum is fp64,
// and p_j = RN(e_j * (1/Z)) with 1/Z carried as two floats, so p_j stays within 2 ulp.
// The host only selects this kernel when smax*|c| <= 80 (no overflow without max subtraction).
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "ptx.cuh"
#include "tile_ops.cuh"

namespace vitint {
namespace {

constexpr int AT_COMPUTE_WARPS = 16;
// Two groups of eight compute warps, or one of sixteen: a query row is shared by 2 or 4 threads, 4 GROUPS warps a TMEM lane quarter.
__host__ __device__ constexpr int at_threads(int groups) { return (AT_COMPUTE_WARPS + groups) * 32; }

struct AttnParams {
    int batch, heads, tokens, q_tiles, total_items;
    int c;                       // container bits of Q, K, V (2 or 4: packed, unpacked in the kernel; 8: one code per byte,
                                 // the TMA copy is the tensor-core operand)
    int n_k;                     // MMA N of Q K^T: tokens rounded up to 16
    int kv_rows;                 // tokens rounded up to 32: K extent of P V, rows of the V tile
    int smax;                    // table covers scores -smax .. smax
    int part_bytes;              // bytes of one of the Q / K / V column blocks in a QKV row
    uint32_t off_table, off_group, group_bytes;         // shared-memory layout
    uint32_t off_pq, off_pk, off_pv, off_q, off_k, off_v, off_p, off_col, off_z, off_mx;   // within a group
    const float* table;          // global copy of the exp table, 2*smax+1 floats
    int at_rest;                 // the table may be read before the grid dependency
    float p_step, p_qp;
    float scale;                 // softmax scale c (GENERAL), c log2 e (SHIFT)
    const float* alpha_o;        // [D]
    const float* beta_o;         // [D] or null
    int out_c;
    float out_qn, out_qp;
    uint8_t* out;
    long long out_pitch;
};

struct AttnBars {
    uint64_t packed_full, v_full, ops_ready, s_full, p_ready, o_full, o_done, grp_sync, z_sync;
};

__global__ void exp_table_kernel(float* table, int smax, float c) {
    grid_dependency_wait();        // an earlier kernel may still read the table
    grid_dependency_launch();
    fill_exp_table(table, smax, c, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// What the compute warps make of the scores: exp from the table; Eq. 4; or exp evaluated per score, for any logits (8-bit codes,
// whose scores are too many to tabulate) -- the arithmetic of softmax_quantize_kernel.
enum AttnMode { AM_TABLE = 0, AM_SHIFT = 1, AM_GENERAL = 2 };

// SHIFT: the softmax of Eq. 4 (2^z with z split into integer part and residual, 2^r ~ 1 + r, integer shifts, the
// division-free comparator quantizer) instead of exp, every step with the result of the stand-alone kernel's integer or
// single fp32 operation, hence the same codes bit for bit.  Two tables of the scores (floor z; the mantissa of 1 + r), 64-bit
// shifts and two comparisons a score took 79 us for 197 tokens x 12 heads at batch 64; computed in pairs, summed in
// doubles and compared only near a tie, 50 us (198 tokens x 6 heads: 42 -> 27).
//
// GROUPS: two pipelines in a CTA, or one with all the warps where no CTA gets a second item.
template <int C, int MODE, int GROUPS>
__global__ void __launch_bounds__(at_threads(GROUPS), 1)
attention_fused_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kv,
                       const __grid_constant__ AttnParams P) {
    static_assert(MODE == AM_TABLE || C == 8, "only the table variant takes packed codes");
    constexpr bool SHIFT = MODE == AM_SHIFT, GENERAL = MODE == AM_GENERAL;
    constexpr int WARPS = AT_COMPUTE_WARPS / GROUPS, H = WARPS / 4;           // compute warps of a group, threads of a row
    extern __shared__ uint8_t smem_raw[];
    __shared__ AttnBars bars[GROUPS];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_addr(smem_raw) + 1023u) & ~1023u;
    uint8_t* const smem_gen = smem_raw + (smem_base - ptx::smem_addr(smem_raw));
    volatile int* abort_ptr = &abort_flag;
    const bool is_control = warp >= AT_COMPUTE_WARPS;
    const int g = is_control ? warp - AT_COMPUTE_WARPS : warp / WARPS;
    AttnBars& B = bars[g];
    const uint32_t gbase = smem_base + P.off_group + (uint32_t)g * P.group_bytes;
    uint8_t* const ggen = smem_gen + P.off_group + (size_t)g * P.group_bytes;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int k = 0; k < GROUPS; ++k) {
            ptx::mbar_init(ptx::smem_addr(&bars[k].packed_full), 1);
            ptx::mbar_init(ptx::smem_addr(&bars[k].v_full), 1);
            ptx::mbar_init(ptx::smem_addr(&bars[k].ops_ready), WARPS);
            ptx::mbar_init(ptx::smem_addr(&bars[k].s_full), 1);
            ptx::mbar_init(ptx::smem_addr(&bars[k].p_ready), WARPS);
            ptx::mbar_init(ptx::smem_addr(&bars[k].o_full), 1);
            ptx::mbar_init(ptx::smem_addr(&bars[k].o_done), WARPS);
            ptx::mbar_init(ptx::smem_addr(&bars[k].grp_sync), WARPS * 32);
            ptx::mbar_init(ptx::smem_addr(&bars[k].z_sync), WARPS);
        }
        ptx::fence_mbar_init();
        ptx::fence_proxy_async_smem();
    }
    if (warp == AT_COMPUTE_WARPS) {                      // first control warp owns the TMEM allocation
        ptx::tmem_alloc(ptx::smem_addr(&tmem_base_slot), GROUPS * 256);
        ptx::tmem_relinquish();
    }
    {
        // P columns behind the last block of eight that holds a token are never written: zero for good
        for (int i = threadIdx.x; i < GROUPS * 128 * 16; i += at_threads(GROUPS)) {
            const int gr = i / 2048, cc = (i >> 7) & 15, r = i & 127;
            if (cc * 16 < P.kv_rows)
                *reinterpret_cast<uint4*>(smem_gen + P.off_group + (size_t)gr * P.group_bytes + P.off_p + (cc >> 3) * 16384 + r * 128 + (((cc & 7) ^ (r & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        ptx::fence_proxy_async_smem();
    }
    if (is_control && lane == 0) { ptx::prefetch_tensormap(&map_q); ptx::prefetch_tensormap(&map_kv); }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // The exp table: global -> shared, once per CTA, while the control warps' first copies and Q K^T are on their way, or before the
    // wait where it cannot come from the kernel in front (the codes do).
    auto table_to_shared = [&]() {
        fill_table_ring(reinterpret_cast<float*>(smem_gen + P.off_table), P.table, P.smax, threadIdx.x, AT_COMPUTE_WARPS * 32);
    };
    if (MODE == AM_TABLE && P.at_rest && !is_control) table_to_shared();
    grid_dependency_wait();
    grid_dependency_launch();
    if constexpr (MODE == AM_TABLE) {
        if (!is_control) {
            if (!P.at_rest) table_to_shared();
            asm volatile("bar.sync 1, %0;" ::"n"(AT_COMPUTE_WARPS * 32) : "memory");
        }
    }
    const uint32_t tmem_grp = __shfl_sync(0xffffffffu, tmem_base_slot, 0) + (uint32_t)g * 256u;

    const int T = P.tokens;
    // Whole waves give every group an item; a remainder of at most one item a CTA goes to one group of as many CTAs as it takes
    // (197 tokens x 12 heads, batch 128: 21 items in the busiest CTA instead of 22, 68.1 -> 65.0 us; batch 1: 24 CTAs instead of
    // 12, 9.2 -> 7.7 us)
    const int wave = gridDim.x * GROUPS, full = P.total_items / wave;
    const int last = full * wave + (P.total_items - full * wave <= (int)gridDim.x ? g * (int)gridDim.x + (int)blockIdx.x
                                                                                  : (int)blockIdx.x * GROUPS + g);
    auto item_at = [&](int n) {                              // the group's n-th item; total_items when there is none
        return n < full ? n * wave + (int)blockIdx.x * GROUPS + g : n == full ? min(last, P.total_items) : P.total_items;
    };
    constexpr bool DIRECT = (C == 8);                  // byte codes: no packed staging, no unpack
    const int head_bytes = 8 * C;                      // 64 codes
    const uint32_t q_bytes = 128u * head_bytes, kv_bytes = (uint32_t)P.kv_rows * head_bytes;   // TMA boxes

    auto item_coords = [&](int item, int& b, int& h, int& qt) {
        const uint32_t two = (uint32_t)P.q_tiles - 1u, bh = (uint32_t)item >> two;           // one or two query tiles
        qt = item & (int)two;
        b = (int)(bh / (uint32_t)P.heads);
        h = (int)bh - b * P.heads;
    };

    if (is_control) {
        // --------------------------- control: TMA + MMA issue ----------------------------
        {
            // packed codes: one barrier for the three slabs, which the compute warps unpack.
            // byte codes: Q and K land in their operand tiles under packed_full, V under v_full, so that each
            // buffer is refilled as soon as the MMA that read it has completed.
            auto issue_loads = [&](int item) {
                int b, h, qt;
                item_coords(item, b, h, qt);
                const uint32_t bar = ptx::smem_addr(&B.packed_full);
                ptx::mbar_arrive_expect_tx(bar, q_bytes + (DIRECT ? 1u : 2u) * kv_bytes);
                ptx::tma_load_3d(gbase + (DIRECT ? P.off_q : P.off_pq), &map_q, bar, h * head_bytes, qt * 128, b);
                ptx::tma_load_3d(gbase + (DIRECT ? P.off_k : P.off_pk), &map_kv, bar, P.part_bytes + h * head_bytes, 0, b);
                if (!DIRECT) ptx::tma_load_3d(gbase + P.off_pv, &map_kv, bar, 2 * P.part_bytes + h * head_bytes, 0, b);
            };
            auto issue_v = [&](int item) {
                int b, h, qt;
                item_coords(item, b, h, qt);
                const uint32_t bar = ptx::smem_addr(&B.v_full);
                ptx::mbar_arrive_expect_tx(bar, kv_bytes);
                ptx::tma_load_3d(gbase + P.off_v, &map_kv, bar, 2 * P.part_bytes + h * head_bytes, 0, b);
            };
            const uint32_t idesc_qk = ptx::idesc_i8(128, P.n_k, 1, 1, 0);
            const uint32_t idesc_pv = ptx::idesc_i8(128, 64, 0, 1, 1);
            const uint64_t q_desc = ptx::smem_desc(gbase + P.off_q, 16, 512, ptx::SWIZZLE_64B);
            const uint64_t k_desc = ptx::smem_desc(gbase + P.off_k, 16, 512, ptx::SWIZZLE_64B);
            const uint64_t v_desc = ptx::smem_desc(gbase + P.off_v, 16, 512, ptx::SWIZZLE_64B);
            const int pv_steps = P.kv_rows / 32;
            bool ok = true;
            int pending = -1, pending_v = -1;       // local index of the item whose loads are in flight
            if (item_at(0) < P.total_items) {
                if (ptx::elect_one()) issue_loads(item_at(0));
                pending = 0;
                if (DIRECT) {
                    if (ptx::elect_one()) issue_v(item_at(0));
                    pending_v = 0;
                }
            }
            for (int n = 0; ok && item_at(n) < P.total_items; ++n) {
                const uint32_t ph = (uint32_t)n & 1u;
                const int next = item_at(n + 1);
                const bool has_next = next < P.total_items;
                if (DIRECT) {
                    if (!mbar_wait_warp(ptx::smem_addr(&B.packed_full), ph, abort_ptr)) { ok = false; break; }
                    pending = -1;
                } else {
                    if (!mbar_wait_warp(ptx::smem_addr(&B.ops_ready), ph, abort_ptr)) { ok = false; break; }
                    pending = -1;
                    if (has_next) {
                        if (ptx::elect_one()) issue_loads(next);
                        pending = n + 1;
                    }
                }
                if (n > 0 && !mbar_wait_warp(ptx::smem_addr(&B.o_done), ph ^ 1u, abort_ptr)) { ok = false; break; }
                ptx::tc_fence_after();
                if (ptx::elect_one()) {
                    for (int k = 0; k < 2; ++k)                    // K = 64 -> two MMAs of 32
                        ptx::mma_i8(tmem_grp, q_desc + (uint64_t)(k * 2), k_desc + (uint64_t)(k * 2), idesc_qk, k);
                    ptx::mma_commit(ptx::smem_addr(&B.s_full));
                }
                __syncwarp();
                if (DIRECT) {
                    // Q K^T has been read out of the Q and K tiles once s_full completes
                    if (!mbar_wait_warp(ptx::smem_addr(&B.s_full), ph, abort_ptr)) { ok = false; break; }
                    if (has_next) {
                        if (ptx::elect_one()) issue_loads(next);
                        pending = n + 1;
                    }
                }
                if (!mbar_wait_warp(ptx::smem_addr(&B.p_ready), ph, abort_ptr)) { ok = false; break; }
                if (DIRECT) {
                    if (!mbar_wait_warp(ptx::smem_addr(&B.v_full), ph, abort_ptr)) { ok = false; break; }
                    pending_v = -1;
                }
                ptx::tc_fence_after();
                if (ptx::elect_one()) {
                    for (int ks = 0; ks < pv_steps; ++ks) {
                        const uint64_t p_desc = ptx::smem_desc(gbase + P.off_p + (uint32_t)(ks >> 2) * 16384u, 16, 1024,
                                                               ptx::SWIZZLE_128B) + (uint64_t)((ks & 3) * 2);
                        ptx::mma_i8(tmem_grp, p_desc, v_desc + (uint64_t)(ks * 128), idesc_pv, ks);
                    }
                    ptx::mma_commit(ptx::smem_addr(&B.o_full));
                }
                __syncwarp();
                if (DIRECT && has_next) {
                    // P V has been read out of the V tile once o_full completes
                    if (!mbar_wait_warp(ptx::smem_addr(&B.o_full), ph, abort_ptr)) { ok = false; break; }
                    if (ptx::elect_one()) issue_v(next);
                    pending_v = n + 1;
                }
            }
            if (!ok) {
                // give the copies still in flight a bounded chance to land before the CTA exits
                if (pending >= 0) {
                    const uint32_t bar = ptx::smem_addr(&B.packed_full);
                    for (int spin = 0; spin < (1 << 20) && !ptx::mbar_try_wait(bar, (uint32_t)pending & 1u); ++spin) {}
                }
                if (pending_v >= 0) {
                    const uint32_t bar = ptx::smem_addr(&B.v_full);
                    for (int spin = 0; spin < (1 << 20) && !ptx::mbar_try_wait(bar, (uint32_t)pending_v & 1u); ++spin) {}
                }
            }
        }
    } else {
        // ------------------------------ compute warps ------------------------------------
        const int wq = warp & 3;                                    // TMEM lane quarter
        const int hf = (warp % WARPS) >> 2;                         // which of the row's H threads: every H-th chunk of 32 columns
        const int tid_g = (warp % WARPS) * 32 + lane;               // within the group
        const int row = wq * 32 + lane;                             // query row of the tile
        double* const zx = reinterpret_cast<double*>(ggen + P.off_z);   // partial row sums, [H][128]
        // An fp64 row sum depends in its last bit on the order of its terms, so both forms keep the same partial sums: pairs of
        // threads `pair` = 0, 1 have the even and the odd chunks, and where a row has four threads the two of a pair share the
        // interleaved sums of one thread of the other form between them.  A row's codes are the same in a batch of any size.
        const int pair = hf & 1, share = hf >> 1;
        auto row_sum = [&]() { return H == 2 ? zx[row] + zx[128 + row] : (zx[row] + zx[256 % (H * 128) + row]) + (zx[128 + row] + zx[384 % (H * 128) + row]); };
        const uint32_t t_row = tmem_grp + ((uint32_t)(wq * 32) << 16);
        const char* const ring = reinterpret_cast<const char*>(smem_gen + P.off_table);
        const uint32_t ring_mask = 8u * (uint32_t)P.smax - 4u;
        float* const colp2 = reinterpret_cast<float*>(ggen + P.off_col);  // alpha[64], beta[64] of the head, one copy per item parity
        const int sh_idx = DIRECT ? 0 : 2 * (8 - C) - 2;            // scaled score -> byte offset 4*S
        const int full_chunks = T >> 5, tail = T & 31, tail_blocks = (tail + 7) >> 3;
        const int tail0 = (hf - full_chunks) & (H - 1);             // the threads with fewer whole chunks take the first blocks of the tail
        const uint32_t qp2 = (uint32_t)P.p_qp * 0x00010001u;
        const bool steep = P.p_step < 1.0f / 65000.0f;              // codes before the clamp might not fit 16 bits
        const double inv_p_step = 1.0 / (double)P.p_step;
        const Divisor p_div = make_divisor(P.p_step);               // (GENERAL)
        bool ok = true;
        for (int n = 0; ok && item_at(n) < P.total_items; ++n) {
            const uint32_t ph = (uint32_t)n & 1u;
            int b, h, qt;
            item_coords(item_at(n), b, h, qt);
            // the head's output parameters; the copy of the other parity may still be read by a warp that is
            // finishing the previous item, and every reader of this one passes z_sync first
            float* const colp = colp2 + (n & 1) * 128;
            if (tid_g < 64) colp[tid_g] = __ldg(P.alpha_o + h * 64 + tid_g);
            else if (tid_g < 128) colp[tid_g] = P.beta_o ? __ldg(P.beta_o + h * 64 + (tid_g - 64)) : 0.0f;
            bool w = true;
            if constexpr (!DIRECT) {
                // ---- operands: packed -> int8 ---------------------------------------------
                w = mbar_wait(ptx::smem_addr(&B.packed_full), ph, abort_ptr);
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                unpack_rows64<C, 1>(ggen + P.off_pq, ggen + P.off_q, 128, tid_g, WARPS * 32);
                unpack_rows64<C, 1>(ggen + P.off_pk, ggen + P.off_k, P.n_k, tid_g, WARPS * 32);
                unpack_rows64<C, 1>(ggen + P.off_pv, ggen + P.off_v, P.kv_rows, tid_g, WARPS * 32);
                ptx::fence_proxy_async_smem();
                ptx::mbar_arrive(ptx::smem_addr(&B.grp_sync));
                w = mbar_wait(ptx::smem_addr(&B.grp_sync), ph, abort_ptr);
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.ops_ready));
            }
            // ---- softmax over the row -------------------------------------------------------
            w = mbar_wait(ptx::smem_addr(&B.s_full), ph, abort_ptr);
            if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
            ptx::tc_fence_after();
            // a warp whose 32 query rows all lie past the last token has nothing to compute: its P rows
            // only feed accumulator rows that are never stored (whatever int8 they hold)
            const bool warp_live = qt * 128 + wq * 32 < T;
            if constexpr (SHIFT || GENERAL) {
                // pass 0: the row's largest score (Eq. 4: the smallest as well).  fl32(S_j c) increases with S_j (c > 0), so the
                // largest score has the largest logit.
                int* const mx = reinterpret_cast<int*>(ggen + P.off_mx);
                int smx = INT_MIN, smn = INT_MAX;
                if (warp_live) {
#pragma unroll 1
                    for (int ch = hf; ch < full_chunks; ch += H) {
                        uint32_t v[32];
                        ptx::tmem_ld32(t_row + (uint32_t)(ch * 32), v);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            smx = max(smx, (int)v[i]);
                            if (SHIFT) smn = min(smn, (int)v[i]);
                        }
                    }
#pragma unroll 1
                    for (int k = tail0; k < tail_blocks; k += H) {
                        uint32_t v[8];
                        ptx::tmem_ld8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            smx = max(smx, 8 * k + i < tail ? (int)v[i] : INT_MIN);
                            if (SHIFT) smn = min(smn, 8 * k + i < tail ? (int)v[i] : INT_MAX);
                        }
                    }
                }
                mx[hf * 128 + row] = smx;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.z_sync));
                w = mbar_wait(ptx::smem_addr(&B.z_sync), 0u, abort_ptr);       // two phases per item: parities 0, 1
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                smx = max(mx[row], mx[128 + row]);
                if constexpr (H == 4) smx = max(smx, max(mx[256 + row], mx[384 + row]));
                const f32x2 c2 = f2_dup(P.scale), nmagic2 = f2_dup(-12582912.0f), magic2 = f2_dup(12582912.0f);
                uint8_t* const prow = ggen + P.off_p + row * 128;
                const int sw = row & 7;
                if constexpr (SHIFT) {
                // pass 1: z_j = fl32(S_j c log2 e), f_j = floor z_j (an addition that rounds down), E_j = trunc((1 + (z_j - f_j)) 2^23)
                // << (30 + f_j - m), m the row's largest f (>> when negative).  While nothing is shifted out, float(E_j) is the float
                // 1 + (z_j - f_j) with 53 + f_j - m added to its exponent; that integer rides in the addend that rounds z_j down.
                // Where the warp's rows spread over at most 21 octaves every E_j is a multiple of 2^9 and a row's sum stays below
                // 2^62, so the 53 bits of a double carry it exactly; otherwise 64-bit integers do.
                const float m = floorf(__fmul_rn((float)smx, P.scale));
                const float addend = 12582912.0f + (53.0f - m);
                const f32x2 add2 = f2_dup(addend), nadd2 = f2_dup(-addend), neg1 = f2_dup(-1.0f), one2 = f2_dup(1.0f);
                auto split = [&](uint32_t a, uint32_t b, f32x2& t, f32x2& r1) {           // t: 1.5 * 2^23 + 53 + f - m; r1: 1 + (z - f)
                    const f32x2 sf = f2_add(f2_pack(__uint_as_float(0x4B400000u + a), __uint_as_float(0x4B400000u + b)), nmagic2);
                    const f32x2 z = f2_mul(sf, c2);
                    t = f2_add_rm(z, add2);
                    r1 = f2_add(f2_fma(f2_add(t, nadd2), neg1, z), one2);
                };
                unsigned long long sigma = 0ull;
                if (warp_live) {
                    const bool wide = floorf(__fmul_rn((float)min(smn, smx), P.scale)) < m - 21.0f;
                    if (!__any_sync(0xffffffffu, wide)) {
                        double zp[2] = {0.0, 0.0};
                        auto term_pair = [&](uint32_t& a, uint32_t& b, bool va, bool vb) {
                            f32x2 t, r1;
                            float t0, t1, x0, x1;
                            split(a, b, t, r1);
                            f2_unpack(t, t0, t1);
                            f2_unpack(r1, x0, x1);
                            a = va ? __float_as_uint(x0) + (__float_as_uint(t0) << 23) : 0u;
                            b = vb ? __float_as_uint(x1) + (__float_as_uint(t1) << 23) : 0u;
                            // the doubles from the bits; a zero becomes 2^-127, which the sum rounds away
                            zp[0] += __hiloint2double((int)((a >> 3) + 0x38000000u), (int)(a << 29));
                            zp[1] += __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
                        };
#pragma unroll 1
                        for (int pc = 2 * hf; pc < 2 * full_chunks; pc += (pc & 1) ? 2 * H - 1 : 1) {     // halves of the thread's chunks
                            uint32_t v[16];
                            ptx::tmem_ld16(t_row + (uint32_t)(pc * 16), v);
                            ptx::tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 16; i += 2) term_pair(v[i], v[i + 1], true, true);
                            ptx::tmem_st16(t_row + (uint32_t)(pc * 16), v);
                        }
#pragma unroll 1
                        for (int k = tail0; k < tail_blocks; k += H) {
                            uint32_t v[8];
                            ptx::tmem_ld8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                            ptx::tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 8; i += 2) term_pair(v[i], v[i + 1], 8 * k + i < tail, 8 * k + i + 1 < tail);
                            ptx::tmem_st8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                        }
                        sigma = (unsigned long long)__double2ll_rn(zp[0] + zp[1]);
                    } else {
                        // the 64-bit term is (M * 2^32) >> (32 - sh) with sh = 30 + f - m kept above -32 (further down everything is
                        // shifted out anyway); what is left of a mantissa shifted right converts by the 2^23 trick
#pragma unroll 1
                        for (int blk = 0; blk < 4 * full_chunks + tail_blocks; ++blk) {           // blocks of eight columns
                            if (blk < 4 * full_chunks ? ((blk >> 2) & (H - 1)) != hf : ((blk - 4 * full_chunks) & (H - 1)) != tail0) continue;
                            uint32_t v[8];
                            ptx::tmem_ld8(t_row + (uint32_t)(blk * 8), v);
                            ptx::tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 8; i += 2) {
                                f32x2 t, r1;
                                float t0, t1, x0, x1;
                                split(v[i], v[i + 1], t, r1);
                                f2_unpack(t, t0, t1);
                                f2_unpack(r1, x0, x1);
#pragma unroll
                                for (int j = 0; j < 2; ++j) {
                                    const bool valid = blk * 8 + i + j < T;
                                    const uint32_t x = __float_as_uint(j ? x1 : x0);
                                    const int sh = max((int)__float_as_uint(j ? t1 : t0) - 0x4B400000 - 23, -31);
                                    const unsigned long long big = ((unsigned long long)(x - 0x3F000000u) << 32) >> (32 - sh);
                                    const uint32_t up = x + ((uint32_t)(sh + 23) << 23);
                                    const uint32_t dn = __float_as_uint(__fadd_rn(__uint_as_float(0x4B000000u + (uint32_t)big), -8388608.0f));
                                    sigma += valid ? big : 0ull;
                                    v[i + j] = valid ? (sh >= 0 ? up : dn) : 0u;
                                }
                            }
                            ptx::tmem_st8(t_row + (uint32_t)(blk * 8), v);
                        }
                    }
                    ptx::tmem_st_wait();
                }
                unsigned long long* const sx = reinterpret_cast<unsigned long long*>(ggen + P.off_z);
                sx[hf * 128 + row] = sigma;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.z_sync));
                w = mbar_wait(ptx::smem_addr(&B.z_sync), 1u, abort_ptr);
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                sigma = sx[row] + sx[128 + row];
                if constexpr (H == 4) sigma += sx[256 + row] + sx[384 + row];
                const float sig_f = __ull2float_rn(sigma);
                // pass 2: the code is the number of references fl32(fl32((k - 1/2) s_P) * Sigma) that float(E_j) exceeds, which is
                // k0 = rint(u), u = min(E_j / (s_P Sigma), Qp), unless u lies next to some k - 1/2: u is off by less than 3.1 units
                // of 2^-24 of itself, a reference by less than 2.1.  An interval of 8 units on either side of u proves a code
                // (197 tokens x 12 heads, batch 64: 44.7 -> 43.5 us against |u - rint(u)| compared with a limit; 198 x 6: 25.5 -> 24.9).
                // Where it does not, values above the last level are kept there for a second look (the first one for a step below
                // 1/65000: 57 us at 1e-5, as at other steps, where comparing all of them took 71), and columns still unproven are
                // compared with the two references around them: k0' = rint(min(u, Qp - 3/4)) is at most one off and never Qp,
                // code = k0' - 1 + [E > ref(k0')] + [E > ref(k0' + 1)], in the float that carries k0' in its mantissa.
                const float inv = warp_live ? __frcp_rn(__fmul_rn(P.p_step, sig_f)) : 0.0f;
                const f32x2 inv2 = f2_dup(inv), lo2 = f2_dup(inv * (1.0f - 4.76837158e-07f)), hi2 = f2_dup(inv * (1.0f + 4.76837158e-07f));
                const float e_top = (P.p_qp + 1.0f) * __fmul_rn(P.p_step, sig_f);
                auto codes = [&](const uint32_t* v, auto& wd, auto count) {
                    constexpr int N = decltype(count)::value;
                    f32x2 e[N / 2];
#pragma unroll
                    for (int i = 0; i < N / 2; ++i) e[i] = f2_pack(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                    if ((steep || __any_sync(0xffffffffu, quantize_interval<N>(e, lo2, hi2, qp2, wd) != 0.0f)) &&
                        __any_sync(0xffffffffu, quantize_interval_below<N>(e, e_top, lo2, hi2, qp2, wd) != 0.0f)) {
                        const float u_top = P.p_qp - 0.75f;
                        const f32x2 half2 = f2_dup(0.5f), nhalf2 = f2_dup(-0.5f), ps2 = f2_dup(P.p_step), sg2 = f2_dup(sig_f);
#pragma unroll
                        for (int i4 = 0; i4 < N / 4; ++i4) {
                            uint32_t cb[4];
#pragma unroll
                            for (int j = 0; j < 4; j += 2) {
                                const float e0 = __uint_as_float(v[4 * i4 + j]), e1 = __uint_as_float(v[4 * i4 + j + 1]);
                                float u0, u1;
                                f2_unpack(f2_mul(f2_pack(e0, e1), inv2), u0, u1);
                                const f32x2 um = f2_add(f2_pack(fminf(u0, u_top), fminf(u1, u_top)), magic2);   // 1.5*2^23 + k0'
                                const f32x2 kf = f2_add(um, nmagic2);
                                float l0, l1, h0, h1;
                                f2_unpack(f2_mul(f2_mul(f2_add(kf, nhalf2), ps2), sg2), l0, l1);
                                f2_unpack(f2_mul(f2_mul(f2_add(kf, half2), ps2), sg2), h0, h1);
                                const f32x2 t_lo = f2_pack(e0 > l0 ? 1.0f : 0.0f, e1 > l1 ? 1.0f : 0.0f);
                                const f32x2 t_hi = f2_pack(e0 > h0 ? 1.0f : 0.0f, e1 > h1 ? 1.0f : 0.0f);
                                float c0, c1;
                                f2_unpack(f2_add(f2_add(um, neg1), f2_add(t_lo, t_hi)), c0, c1);
                                cb[j] = __float_as_uint(c0);
                                cb[j + 1] = __float_as_uint(c1);
                            }
                            wd[i4] = __byte_perm(__byte_perm(cb[0], cb[1], 0x4040), __byte_perm(cb[2], cb[3], 0x4040), 0x5410);
                        }
                    }
                };
                if (warp_live) {
#pragma unroll 1
                    for (int pc = 2 * hf; pc < 2 * full_chunks; pc += (pc & 1) ? 2 * H - 1 : 1) {
                        uint32_t v[16], wd[4];
                        ptx::tmem_ld16(t_row + (uint32_t)(pc * 16), v);
                        ptx::tmem_ld_wait();
                        codes(v, wd, std::integral_constant<int, 16>{});
                        *reinterpret_cast<uint4*>(prow + (pc >> 3) * 16384 + (((pc & 7) ^ sw) << 4)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                    }
#pragma unroll 1
                    for (int k = tail0; k < tail_blocks; k += H) {
                        uint32_t v[8], wd[2];
                        const int col = full_chunks * 32 + k * 8, cc = col >> 4;
                        ptx::tmem_ld8(t_row + (uint32_t)col, v);
                        ptx::tmem_ld_wait();
                        codes(v, wd, std::integral_constant<int, 8>{});
                        *reinterpret_cast<uint2*>(prow + (cc >> 3) * 16384 + (((cc & 7) ^ sw) << 4) + (col & 8)) = make_uint2(wd[0], wd[1]);
                    }
                }
                } else {
                // exp(t_j - max) by reduction and polynomial, row sum in fp64, p = e / Z with 1/Z as two floats, one exact division
                // by s_P
                const f32x2 nmx2 = f2_dup(-__fmul_rn((float)smx, P.scale));
                double zp[H == 2 ? 2 : 1] = {};
                auto exp_pair = [&](uint32_t& a, uint32_t& b, bool va, bool vb) {
                    const f32x2 sf = f2_add(f2_pack(__uint_as_float(0x4B400000u + a), __uint_as_float(0x4B400000u + b)), nmagic2);   // |S| <= 2^20
                    float e0, e1;
                    f2_unpack(exp_reduced2(f2_mul(sf, c2), nmx2), e0, e1);
                    a = va ? __float_as_uint(e0) : 0u;
                    b = vb ? __float_as_uint(e1) : 0u;
                    // the doubles from the bits; a zero becomes 2^-127, which a sum of at least 1 does not see
                    zp[0] += __hiloint2double((int)((a >> 3) + 0x38000000u), (int)(a << 29));
                    zp[H == 2 ? 1 : 0] += __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
                };
                if (H == 4 && warp_live) {
                    // a thread of two in place of one that has the chunk in the other form: the even or the odd columns
                    const uint32_t t_own = t_row + (uint32_t)share;
#pragma unroll 1
                    for (int pc = 2 * pair; pc < 2 * full_chunks; pc += (pc & 1) ? 3 : 1) {           // halves of the pair's chunks
                        uint32_t v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) ptx::tmem_ld1(t_own + (uint32_t)(pc * 16 + 2 * i), v[i]);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; i += 2) exp_pair(v[i], v[i + 1], true, true);
#pragma unroll
                        for (int i = 0; i < 8; ++i) ptx::tmem_st1(t_own + (uint32_t)(pc * 16 + 2 * i), v[i]);
                    }
#pragma unroll 1
                    for (int k = (pair - full_chunks) & 1; k < tail_blocks; k += 2) {
                        const uint32_t t_blk = t_own + (uint32_t)(full_chunks * 32 + k * 8);
                        uint32_t v[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) ptx::tmem_ld1(t_blk + (uint32_t)(2 * i), v[i]);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 4; i += 2) exp_pair(v[i], v[i + 1], 8 * k + 2 * i + share < tail, 8 * k + 2 * i + 2 + share < tail);
#pragma unroll
                        for (int i = 0; i < 4; ++i) ptx::tmem_st1(t_blk + (uint32_t)(2 * i), v[i]);
                    }
                    ptx::tmem_st_wait();
                }
                if (H == 2 && warp_live) {
#pragma unroll 1
                    for (int pc = 2 * hf; pc < 2 * full_chunks; pc += (pc & 1) ? 3 : 1) {             // halves of the thread's chunks
                        uint32_t v[16];
                        ptx::tmem_ld16(t_row + (uint32_t)(pc * 16), v);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; i += 2) exp_pair(v[i], v[i + 1], true, true);
                        ptx::tmem_st16(t_row + (uint32_t)(pc * 16), v);
                    }
#pragma unroll 1
                    for (int k = tail0; k < tail_blocks; k += H) {
                        uint32_t v[8];
                        ptx::tmem_ld8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 8; i += 2) exp_pair(v[i], v[i + 1], 8 * k + i < tail, 8 * k + i + 1 < tail);
                        ptx::tmem_st8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                    }
                    ptx::tmem_st_wait();
                }
                zx[hf * 128 + row] = H == 2 ? zp[0] + zp[H == 2 ? 1 : 0] : zp[0];
                if constexpr (H == 4) ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.z_sync));
                w = mbar_wait(ptx::smem_addr(&B.z_sync), 1u, abort_ptr);
                if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
                if constexpr (H == 4) ptx::tc_fence_after();         // pass 2 reads exponentials that other warps have stored
                const double z = row_sum();
                const double r0 = (double)__frcp_rn((float)z), rz = r0 * (2.0 - z * r0);
                const float rzh = (float)rz, rzl = (float)(rz - (double)(float)rz);
                const f32x2 rzh2 = f2_dup(rzh), rzl2 = f2_dup(rzl), dr2 = f2_dup(p_div.r), ndb2 = f2_dup(-p_div.b);
                // two roundings separate the definition's argument from e / (Z s_P); within 2.1 units of 2^-24 codes are proven (the
                // division itself costs five packed operations a pair: a layer of 8-bit codes at batch 32, 120.1 -> 118.9 us)
                const double rs = rz * inv_p_step;
                const f32x2 lo2 = f2_dup(__double2float_rd(rs * (1.0 - 2.1 / 16777216.0))), hi2 = f2_dup(__double2float_ru(rs * (1.0 + 2.1 / 16777216.0)));
                const bool doubt = steep || !((float)rs > 1e-37f);
                auto code_pair = [&](uint32_t a, uint32_t b) -> uint32_t {                     // two codes in 16-bit halves
                    const f32x2 e = f2_pack(__uint_as_float(a), __uint_as_float(b));
                    const f32x2 p = f2_fma(e, rzh2, f2_mul(e, rzl2));
                    float q0, q1, c0, c1;
                    if (p_div.exact) {
                        const f32x2 qa = f2_mul(p, dr2);                                       // Markstein: RN(p / step) in three operations
                        f2_unpack(f2_fma(f2_fma(qa, ndb2, p), dr2, qa), q0, q1);
                    } else {
                        f2_unpack(p, q0, q1);
                        q0 = __fdiv_rn(q0, p_div.b);
                        q1 = __fdiv_rn(q1, p_div.b);
                    }
                    f2_unpack(f2_add(f2_pack(fminf(q0, P.p_qp), fminf(q1, P.p_qp)), magic2), c0, c1);
                    return __byte_perm(__float_as_uint(c0), __float_as_uint(c1), 0x5410);
                };
                auto codes = [&](const uint32_t* v, auto& wd, auto count) {
                    constexpr int N = decltype(count)::value;
                    f32x2 e[N / 2];
#pragma unroll
                    for (int i = 0; i < N / 2; ++i) e[i] = f2_pack(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                    if (__any_sync(0xffffffffu, quantize_interval<N>(e, lo2, hi2, qp2, wd) != 0.0f || doubt)) {
#pragma unroll
                        for (int i = 0; i < N / 4; ++i)
                            wd[i] = __byte_perm(code_pair(v[4 * i], v[4 * i + 1]), code_pair(v[4 * i + 2], v[4 * i + 3]), 0x6420);
                    }
                };
                if (warp_live) {
#pragma unroll 1
                    for (int pc = 2 * hf; pc < 2 * full_chunks; pc += (pc & 1) ? 2 * H - 1 : 1) {
                        uint32_t v[16], wd[4];
                        ptx::tmem_ld16(t_row + (uint32_t)(pc * 16), v);
                        ptx::tmem_ld_wait();
                        codes(v, wd, std::integral_constant<int, 16>{});
                        *reinterpret_cast<uint4*>(prow + (pc >> 3) * 16384 + (((pc & 7) ^ sw) << 4)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                    }
#pragma unroll 1
                    for (int k = tail0; k < tail_blocks; k += H) {
                        uint32_t v[8], wd[2];
                        const int col = full_chunks * 32 + k * 8, cc = col >> 4;
                        ptx::tmem_ld8(t_row + (uint32_t)col, v);
                        ptx::tmem_ld_wait();
                        codes(v, wd, std::integral_constant<int, 8>{});
                        *reinterpret_cast<uint2*>(prow + (cc >> 3) * 16384 + (((cc & 7) ^ sw) << 4) + (col & 8)) = make_uint2(wd[0], wd[1]);
                    }
                }
                }   // Eq. 4 / exp per score
            } else {
            // pass 1: e_j = EXP[S_j], row sum in fp64, e_j parked in TMEM over S_j; whole chunks of 32 columns, then the tail
            // by blocks of eight (197 tokens: 200 columns walked instead of 224)
            double zsum = 0.0;
            if (warp_live) {
                uint32_t v0[16], v1[16];
                if constexpr (H == 2) {
                    // sixteen columns are looked up while the next sixteen are on their way
                    double zp[4] = {0.0, 0.0, 0.0, 0.0};
                    if (hf < full_chunks) ptx::tmem_ld16(t_row + (uint32_t)(hf * 32), v0);
#pragma unroll 1
                    for (int ch = hf; ch < full_chunks; ch += H) {
                        const uint32_t t_ch = t_row + (uint32_t)(ch * 32);
                        ptx::tmem_ld_wait();
                        ptx::tmem_ld16(t_ch + 16, v1);
                        exp_lookup<16, !DIRECT, false>(v0, ring, ring_mask, sh_idx, 16, zp);
                        ptx::tmem_st16(t_ch, v0);
                        ptx::tmem_ld_wait();
                        if (ch + H < full_chunks) ptx::tmem_ld16(t_ch + 32 * H, v0);
                        exp_lookup<16, !DIRECT, false>(v1, ring, ring_mask, sh_idx, 16, zp);
                        ptx::tmem_st16(t_ch + 16, v1);
                    }
#pragma unroll 1
                    for (int k = tail0; k < tail_blocks; k += H) {
                        uint32_t v[8];
                        ptx::tmem_ld8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                        ptx::tmem_ld_wait();
                        exp_lookup<8, !DIRECT, true>(v, ring, ring_mask, sh_idx, tail - 8 * k, zp);
                        ptx::tmem_st8(t_row + (uint32_t)(full_chunks * 32 + k * 8), v);
                    }
                    zsum = (zp[0] + zp[1]) + (zp[2] + zp[3]);
                } else {
                    // a thread of two in place of one that has the chunk in the other form: two of every four columns
                    double zp[2] = {0.0, 0.0};
                    const uint32_t t_own = t_row + (uint32_t)(2 * share);
                    auto load = [&](int ch, uint32_t (&v)[16]) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) ptx::tmem_ld2(t_own + (uint32_t)(ch * 32 + 4 * i), v[2 * i], v[2 * i + 1]);
                    };
                    auto entries = [&](int ch, uint32_t (&v)[16]) {
                        exp_lookup<16, !DIRECT, false>(v, ring, ring_mask, sh_idx, 32, zp);
#pragma unroll
                        for (int i = 0; i < 8; ++i) ptx::tmem_st2(t_own + (uint32_t)(ch * 32 + 4 * i), v[2 * i], v[2 * i + 1]);
                    };
                    if (pair < full_chunks) load(pair, v0);
#pragma unroll 1
                    for (int ch = pair; ch < full_chunks; ch += 4) {
                        ptx::tmem_ld_wait();
                        if (ch + 2 < full_chunks) load(ch + 2, v1);
                        entries(ch, v0);
                        if (ch + 2 < full_chunks) {
                            ptx::tmem_ld_wait();
                            if (ch + 4 < full_chunks) load(ch + 4, v0);
                            entries(ch + 2, v1);
                        }
                    }
#pragma unroll 1
                    for (int k = (pair - full_chunks) & 1; k < tail_blocks; k += 2) {
                        const uint32_t t_blk = t_own + (uint32_t)(full_chunks * 32 + k * 8);
                        uint32_t v[4];
                        ptx::tmem_ld2(t_blk, v[0], v[1]);
                        ptx::tmem_ld2(t_blk + 4, v[2], v[3]);
                        ptx::tmem_ld_wait();
                        exp_lookup<4, !DIRECT, true>(v, ring, ring_mask, sh_idx, tail - 8 * k - 2 * share, zp);
                        ptx::tmem_st2(t_blk, v[0], v[1]);
                        ptx::tmem_st2(t_blk + 4, v[2], v[3]);
                    }
                    zsum = zp[0] + zp[1];
                }
                ptx::tmem_st_wait();
            }
            // the row's threads add their partial sums (every warp takes part in the barrier)
            zx[hf * 128 + row] = zsum;
            if constexpr (H == 4) ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.z_sync));
            w = mbar_wait(ptx::smem_addr(&B.z_sync), ph, abort_ptr);
            if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
            if constexpr (H == 4) ptx::tc_fence_after();             // pass 2 reads entries that other warps have stored
            const double z = row_sum();
            // r = 1 / (Z * s_P) as a two-float number: e * r then carries the quantizer argument p / s_P to
            // about half an ulp, i.e. it is the exact-division result for a probability that differs from
            // RN(e / Z) by less than one ulp
            const double rz = warp_live ? inv_p_step / z : 0.0;
            const float rzh = (float)rz;
            const float rzl = (float)(rz - (double)rzh);
            const f32x2 rzh2 = f2_dup(rzh), rzl2 = f2_dup(rzl);
            uint8_t* const prow = ggen + P.off_p + row * 128;
            const int sw = row & 7;
            // pass 2: code = min(rint(e_j / (Z s_P)), Qp) (p >= 0: no lower clamp)
            if (warp_live) {
                const float e_top = steep ? 60000.0f / rzh : 0.0f;         // far above Qp, below 2^16
#pragma unroll 1
                for (int ch = hf; ch < full_chunks; ch += H) {
                    uint32_t v[32], wd[8];
                    ptx::tmem_ld32(t_row + (uint32_t)(ch * 32), v);
                    ptx::tmem_ld_wait();
                    if (steep) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(fminf(__uint_as_float(v[i]), e_top));
                    }
                    quantize_entries<32>(v, rzh2, rzl2, qp2, wd);
                    // 32 codes = two 16-byte chunks cc = 2*ch, 2*ch+1 of this row's 256-byte K extent
                    const int cc = 2 * ch;
                    uint8_t* const blk = prow + (cc >> 3) * 16384;
                    *reinterpret_cast<uint4*>(blk + (((cc & 7) ^ sw) << 4)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                    *reinterpret_cast<uint4*>(blk + ((((cc + 1) & 7) ^ sw) << 4)) = make_uint4(wd[4], wd[5], wd[6], wd[7]);
                }
#pragma unroll 1
                for (int k = tail0; k < tail_blocks; k += H) {
                    uint32_t v[8], wd[2];
                    const int col = full_chunks * 32 + k * 8, cc = col >> 4;
                    ptx::tmem_ld8(t_row + (uint32_t)col, v);
                    ptx::tmem_ld_wait();
                    if (steep) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = __float_as_uint(fminf(__uint_as_float(v[i]), e_top));
                    }
                    quantize_entries<8>(v, rzh2, rzl2, qp2, wd);
                    *reinterpret_cast<uint2*>(prow + (cc >> 3) * 16384 + (((cc & 7) ^ sw) << 4) + (col & 8)) = make_uint2(wd[0], wd[1]);
                }
            }
            }
            ptx::fence_proxy_async_smem();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.p_ready));
            // ---- O = P V: requantize and store ------------------------------------------------
            w = mbar_wait(ptx::smem_addr(&B.o_full), ph, abort_ptr);
            if (!__all_sync(0xffffffffu, w)) { ok = false; break; }
            ptx::tc_fence_after();
            const int token = qt * 128 + row;
            // each of the row's threads requantizes and stores its share of the head's 64 columns (V codes that were unpacked sit
            // in the high bits of their bytes)
            if (warp_live) {
                constexpr int N = 64 / H;
                uint32_t v[N], ow[N / 4];
                if constexpr (H == 2) ptx::tmem_ld32(t_row + (uint32_t)(hf * N), v);
                else ptx::tmem_ld16(t_row + (uint32_t)(hf * N), v);
                ptx::tmem_ld_wait();
                requantize_row<!GENERAL, N>(v, 8 - C, colp + hf * N, colp + 64 + hf * N, P.out_qn, P.out_qp, ow);
                if (token < T)
                    store_row(P.out + ((long long)b * T + token) * P.out_pitch + (long long)h * (8 * P.out_c) + hf * (N * P.out_c / 8), ow, P.out_c);
            }
            // row padding behind the last head's columns (a caller may choose a pitch beyond the row's codes)
            if (token < T && h == P.heads - 1 && hf == H - 1) {
                uint8_t* const orow = P.out + ((long long)b * T + token) * P.out_pitch;
                for (long long off = (long long)P.heads * (8 * P.out_c); off + 4 <= P.out_pitch; off += 4)
                    *reinterpret_cast<uint32_t*>(orow + off) = 0u;
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&B.o_done));
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == AT_COMPUTE_WARPS) {
        ptx::tc_fence_after();
        __syncwarp();
        ptx::tmem_dealloc(tmem_base_slot, GROUPS * 256);
    }
}

inline uint32_t up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

}  // namespace
}  // namespace vitint

using namespace vitint;

extern "C" size_t vitint_attention_core_shift_workspace_bytes(int32_t bits) {
    if (bits != 2 && bits != 3 && bits != 4) return 0;
    const int m = 1 << (container_bits(bits) - 1);
    return (size_t)(2 * 64 * m * m + 2) * 6 + 256;                   // six bytes a score: what the contract has asked for since the kernel kept tables
}

extern "C" size_t vitint_attention_core_workspace_bytes(int32_t bits) {
    if (bits != 2 && bits != 3 && bits != 4) return 0;
    const int m = 1 << (container_bits(bits) - 1);   // sized by the container: any bit pattern indexes inside
    return (size_t)(2 * 64 * m * m + 1) * sizeof(float) + 256;
}

namespace vitint {
int attention_long_launch(const vitint_codes* qkv, int batch, int heads, int tokens, int smax, const float* table, float cs, float p_step,
                          float p_qp, const float* alpha_o, const float* beta_o, const vitint_codes* o_out, cudaStream_t st);
}

// Shared by the three entry points below.  build_table: fill `workspace` with the exp table first (one more
// small launch); otherwise the caller has filled it for exactly these steps and bits (vitint_attention_exp_table).
static int attention_core_launch(const vitint_codes* qkv, int32_t batch, int32_t heads, int32_t tokens,
                                 float q_step, float k_step, float p_step, int32_t p_bits, const float* alpha_o,
                                 const float* beta_o, const vitint_codes* o_out, void* workspace,
                                 size_t workspace_bytes, bool build_table, void* stream, int mode = AM_TABLE) {
    const bool shift = mode == AM_SHIFT, general = mode == AM_GENERAL;
    if (int rc = check_codes(qkv)) return rc;
    if (int rc = check_codes(o_out)) return rc;
    if (batch <= 0 || heads <= 0 || tokens <= 0 || !alpha_o) return VITINT_ERR_INVALID_ARG;
    const int64_t M = (int64_t)batch * tokens, D = (int64_t)heads * 64;
    if (qkv->rows != M || qkv->cols != 3 * D || !qkv->is_signed || o_out->rows != M || o_out->cols != D)
        return VITINT_ERR_INVALID_ARG;
    const float steps[3] = {q_step, k_step, p_step};
    for (float s : steps) if (!(s > 0.0f && s < INFINITY)) return VITINT_ERR_INVALID_ARG;
    if (!valid_bits(p_bits)) return VITINT_ERR_INVALID_ARG;
    if ((qkv->bits == 8 && !general) || batch > 65535) return VITINT_ERR_UNSUPPORTED;
    const int c = codes_container(qkv);                  // 2 / 4: packed; 8: one code per byte
    // beyond 256 tokens S no longer fits tensor memory beside O: the chunked two-pass kernel (byte-stored codes, exp table)
    const bool long_seq = tokens > 256;
    if (long_seq && (mode != AM_TABLE || c != 8 || tokens > 4096)) return VITINT_ERR_UNSUPPORTED;
    if (general && c != 8) return VITINT_ERR_UNSUPPORTED;
    const int m = 1 << (container_bits(qkv->bits) - 1);
    const int smax = 64 * m * m;
    const float cs = (float)((double)q_step * (double)k_step / 8.0);
    // exp without max subtraction must not overflow for any score the declared code range can produce
    // (the table itself is sized by the container so that any bit pattern indexes inside it)
    const int mq = 1 << (qkv->bits - 1);
    if (mode == AM_TABLE && 64.0 * mq * mq * (double)cs > 80.0) return VITINT_ERR_UNSUPPORTED;
    // Eq. 4: z = S * c2 with c2 = c * log2 e; the row maximum is subtracted (as shifts), so the only range limit is that floor z
    // is added in the integers between 2^23 and 2^24.  Byte-stored codes only.
    const float c2 = (float)((double)cs * 1.4426950408889634);
    if (shift && (c != 8 || (double)smax * (double)c2 > 30000.0)) return VITINT_ERR_UNSUPPORTED;
    if (!general && (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) ||
        workspace_bytes < (shift ? vitint_attention_core_shift_workspace_bytes(qkv->bits)
                                 : vitint_attention_core_workspace_bytes(qkv->bits))))
        return VITINT_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    if (long_seq) {
        if (build_table) {
            launch_kernel(exp_table_kernel, dim3((2 * smax + 1 + 255) / 256), dim3(256), 0, st, (float*)workspace, smax, cs);
            if (cudaGetLastError() != cudaSuccess) return VITINT_ERR_CUDA;
        }
        int pqn, pqp;
        code_range(p_bits, 0, &pqn, &pqp);
        return attention_long_launch(qkv, batch, heads, tokens, smax, (const float*)workspace, cs, p_step, (float)pqp, alpha_o,
                                     beta_o, o_out, st);
    }

    AttnParams P{};
    P.batch = batch; P.heads = heads; P.tokens = tokens;
    P.q_tiles = (tokens + 127) / 128;
    P.total_items = batch * heads * P.q_tiles;
    P.c = c;
    P.n_k = (tokens + 15) / 16 * 16;
    P.kv_rows = (tokens + 31) / 32 * 32;
    P.smax = smax;
    P.scale = shift ? c2 : cs;
    P.part_bytes = (int)(D * c / 8);
    P.table = (const float*)workspace;
    P.at_rest = parameters_at_rest() && !build_table ? 1 : 0;
    P.p_step = p_step;
    int qn, qp;
    code_range(p_bits, 0, &qn, &qp);
    P.p_qp = (float)qp;
    P.alpha_o = alpha_o; P.beta_o = beta_o;
    P.out_c = codes_container(o_out);
    code_range(o_out->bits, o_out->is_signed, &qn, &qp);
    P.out_qn = (float)qn; P.out_qp = (float)qp;
    P.out = (uint8_t*)o_out->data; P.out_pitch = o_out->pitch_bytes;
    // shared-memory layout
    const uint32_t hb = 8u * c;
    P.off_table = 0;
    P.off_group = mode != AM_TABLE ? 0u : up((uint32_t)(2 * smax + 1) * 4u, 1024);
    uint32_t o = 0;
    P.off_q = o; o += 128 * 64;
    P.off_k = o; o += up((uint32_t)(c == 8 ? P.kv_rows : P.n_k) * 64, 1024);   // byte codes: the K box is kv_rows high
    P.off_v = o; o += up((uint32_t)P.kv_rows * 64, 1024);
    P.off_p = o; o += (uint32_t)((P.kv_rows + 127) / 128) * 16384u;
    if (c != 8) {
        P.off_pq = o; o += up(128 * hb, 128);
        P.off_pk = o; o += up((uint32_t)P.kv_rows * hb, 128);
        P.off_pv = o; o += up((uint32_t)P.kv_rows * hb, 128);
    }
    P.off_col = o; o += 1024;
    // One group of sixteen warps where every item has a CTA of its own: with two groups of eight the other half of the warps has
    // nothing to do.  197 tokens x 12 heads, one image, inside a stack of layers: 7.9 -> 6.2 us together with the copies
    // of Q, K and V being under way while the exp table is filled (192 items on 96 CTAs of two groups, 9.3 -> 7.4 by the latter).
    const int sms = sm_count(), groups = P.total_items <= sms ? 1 : 2, row_threads = 4 / groups;
    P.off_z = o; o += row_threads * 128 * 8;
    P.off_mx = o;
    if (mode != AM_TABLE) o += row_threads * 128 * 4;      // partial row maxima
    P.group_bytes = up(o, 1024);
    const size_t smem = (size_t)P.off_group + (size_t)groups * P.group_bytes + 1024;
    if (smem > 225 * 1024) return VITINT_ERR_UNSUPPORTED;

    CUtensorMap map_q, map_kv;
    {
        // 3-D byte view of the QKV code matrix: (row bytes, token, image); rows past an image's
        // last token read as zero.  Q tiles are 128 rows high, K and V tiles kv_rows.
        EncodeTiledFn fn = encode_fn();
        if (!fn) return VITINT_ERR_CUDA;
        cuuint64_t dims[3] = {(cuuint64_t)codes_row_bytes(qkv, 3 * D), (cuuint64_t)tokens, (cuuint64_t)batch};
        // byte codes land directly in the 64-byte-swizzled operand tiles
        const CUtensorMapSwizzle swz = c == 8 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE;
        cuuint64_t strides[2] = {(cuuint64_t)qkv->pitch_bytes, (cuuint64_t)qkv->pitch_bytes * tokens};
        cuuint32_t estr[3] = {1, 1, 1};
        cuuint32_t box_q[3] = {hb, 128, 1}, box_kv[3] = {hb, (cuuint32_t)P.kv_rows, 1};
        if (fn(&map_q, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, qkv->data, dims, strides, box_q, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
            fn(&map_kv, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, qkv->data, dims, strides, box_kv, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return VITINT_ERR_CUDA;
    }
    if (build_table && mode == AM_TABLE) {
        launch_kernel(exp_table_kernel, dim3((2 * smax + 1 + 255) / 256), dim3(256), 0, st, (float*)workspace, smax, cs);
        if (cudaGetLastError() != cudaSuccess) return VITINT_ERR_CUDA;
    }
    int grid = sms;
    if (grid >= P.total_items) grid = P.total_items;                         // one item a CTA
    else if (grid > (P.total_items + 1) / 2) grid = (P.total_items + 1) / 2; // one item a group
    const int dev = current_device();
    if (dev < 0) return VITINT_ERR_CUDA;
    static bool attr_set[MAX_DEVICES][10] = {};
    auto launch = [&](auto kernel, int slot) -> int {
        if (!attr_set[dev][slot]) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024) != cudaSuccess) return VITINT_ERR_CUDA;
            attr_set[dev][slot] = true;
        }
        launch_kernel(kernel, dim3(grid), dim3(at_threads(groups)), smem, st, map_q, map_kv, P);
        return cuda_status(cudaGetLastError());
    };
    auto by_mode = [&](auto g) -> int {
        constexpr int G = decltype(g)::value, s0 = 5 * (G - 1);
        if (general) return launch(attention_fused_kernel<8, AM_GENERAL, G>, s0 + 4);
        if (shift) return launch(attention_fused_kernel<8, AM_SHIFT, G>, s0 + 3);
        if (c == 8) return launch(attention_fused_kernel<8, AM_TABLE, G>, s0 + 2);
        if (c == 4) return launch(attention_fused_kernel<4, AM_TABLE, G>, s0 + 1);
        return launch(attention_fused_kernel<2, AM_TABLE, G>, s0);
    };
    return groups == 1 ? by_mode(std::integral_constant<int, 1>{}) : by_mode(std::integral_constant<int, 2>{});
}

extern "C" int vitint_attention_core(const vitint_codes* qkv, int32_t batch, int32_t heads, int32_t tokens,
                                     float q_step, float k_step, float p_step, int32_t p_bits, const float* alpha_o,
                                     const float* beta_o, const vitint_codes* o_out, void* workspace,
                                     size_t workspace_bytes, void* stream) {
    return attention_core_launch(qkv, batch, heads, tokens, q_step, k_step, p_step, p_bits, alpha_o, beta_o, o_out,
                                 workspace, workspace_bytes, true, stream);
}

namespace vitint {
// The fused core for logits of any range (no table, no workspace), byte-stored codes up to 8 bits and 256 tokens; the codes of
// P are those of vitint_softmax_quantize.  197 tokens x 12 heads of 8-bit codes, batch 32: 34 us, against 87 us as
// Q K^T, softmax and P V with S and P in memory.
int attention_core_general(const vitint_codes* qkv, int batch, int heads, int tokens, float q_step, float k_step, float p_step,
                           int p_bits, const float* alpha_o, const float* beta_o, const vitint_codes* o_out, void* stream) {
    return attention_core_launch(qkv, batch, heads, tokens, q_step, k_step, p_step, p_bits, alpha_o, beta_o, o_out, nullptr, 0, false,
                                 stream, AM_GENERAL);
}
}  // namespace vitint

extern "C" int vitint_attention_core_shift(const vitint_codes* qkv, int32_t batch, int32_t heads, int32_t tokens,
                                           float q_step, float k_step, float p_step, int32_t p_bits, const float* alpha_o,
                                           const float* beta_o, const vitint_codes* o_out, void* workspace,
                                           size_t workspace_bytes, int32_t table_ready, void* stream) {
    return attention_core_launch(qkv, batch, heads, tokens, q_step, k_step, p_step, p_bits, alpha_o, beta_o, o_out,
                                 workspace, workspace_bytes, table_ready == 0, stream, AM_SHIFT);
}

extern "C" int vitint_attention_exp_table(int32_t bits, float q_step, float k_step, void* table, size_t table_bytes,
                                          void* stream) {
    if (!valid_bits(bits) || bits == 8) return VITINT_ERR_UNSUPPORTED;
    if (!(q_step > 0.0f && q_step < INFINITY) || !(k_step > 0.0f && k_step < INFINITY)) return VITINT_ERR_INVALID_ARG;
    if (!table || (reinterpret_cast<uintptr_t>(table) & 255u) || table_bytes < vitint_attention_core_workspace_bytes(bits))
        return VITINT_ERR_WORKSPACE;
    const int m = 1 << (container_bits(bits) - 1);
    const int smax = 64 * m * m;
    const float cs = (float)((double)q_step * (double)k_step / 8.0);
    launch_kernel(exp_table_kernel, dim3((2 * smax + 1 + 255) / 256), dim3(256), 0, (cudaStream_t)stream, (float*)table,
                  smax, cs);
    return cuda_status(cudaGetLastError());
}

extern "C" int vitint_attention_core_prepared(const vitint_codes* qkv, int32_t batch, int32_t heads, int32_t tokens,
                                              float q_step, float k_step, float p_step, int32_t p_bits,
                                              const float* alpha_o, const float* beta_o, const vitint_codes* o_out,
                                              const void* table, size_t table_bytes, void* stream) {
    return attention_core_launch(qkv, batch, heads, tokens, q_step, k_step, p_step, p_bits, alpha_o, beta_o, o_out,
                                 const_cast<void*>(table), table_bytes, false, stream);
}

// ---------------------------------------------------------------------------------------
// Allocation-free variant: the exp table lives in a fixed device array of this library.
// ---------------------------------------------------------------------------------------
namespace vitint {
namespace {

constexpr int STATIC_TABLE_FLOATS = 8320;   // largest table (8193 entries, 4-bit containers) plus the 256-byte slack of the workspace query

// Resident on every GPU that loads the library, from load until the process exits (about 33 KB).
static __device__ __align__(256) float g_static_exp_table[STATIC_TABLE_FLOATS];

// the widest codes the table-driven kernel takes (4-bit containers: scores in -4096 .. 4096) must fit the array
static_assert((2 * 64 * 8 * 8 + 1) * sizeof(float) + 256 <= sizeof(float) * STATIC_TABLE_FLOATS,
              "the built-in scratch must hold the exp table of 4-bit codes");

void* g_static_table_addr[MAX_DEVICES];   // device address of the array, per device, once looked up
int g_static_table_rc[MAX_DEVICES];
std::once_flag g_static_table_once[MAX_DEVICES];

// The array's name is only a host-side handle; kernels need its device address.  Looked up once
// per device, with that device current (std::call_once: concurrent first calls from several host
// threads are safe).
int static_table_address(void** out) {
    const int dev = current_device();
    if (dev < 0) return VITINT_ERR_CUDA;
    std::call_once(g_static_table_once[dev], [dev]() {
        void* p = nullptr;
        const bool ok = cudaGetSymbolAddress(&p, g_static_exp_table) == cudaSuccess && p != nullptr;
        g_static_table_addr[dev] = ok ? p : nullptr;
        g_static_table_rc[dev] = ok ? VITINT_OK : VITINT_ERR_CUDA;
    });
    if (g_static_table_rc[dev] != VITINT_OK) return g_static_table_rc[dev];
    *out = g_static_table_addr[dev];
    return VITINT_OK;
}

}  // namespace
}  // namespace vitint

extern "C" int vitint_attention_core_noalloc(const vitint_codes* qkv, int32_t batch, int32_t heads, int32_t tokens,
                                             float q_step, float k_step, float p_step, int32_t p_bits,
                                             const float* alpha_o, const float* beta_o, const vitint_codes* o_out,
                                             void* stream) {
    // argument errors first, so that they are reported exactly as vitint_attention_core reports them
    if (int rc = check_codes(qkv)) return rc;
    if (int rc = check_codes(o_out)) return rc;
    const size_t need = vitint_attention_core_workspace_bytes(qkv->bits);
    if (need == 0) return VITINT_ERR_UNSUPPORTED;                     // 8-bit codes: no table-driven kernel
    void* table = nullptr;
    if (int rc = static_table_address(&table)) return rc;
    return vitint_attention_core(qkv, batch, heads, tokens, q_step, k_step, p_step, p_bits, alpha_o, beta_o, o_out,
                                 table, sizeof(float) * STATIC_TABLE_FLOATS, stream);
}

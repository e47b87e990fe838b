// a4 + a5 + a6 fused for sequences beyond 256 tokens (577, 785: S no longer fits tensor memory beside O).
//
// Per (image, head, 128-query tile) the keys are walked in chunks of at most 192, twice:
//   pass A   S_c = Q K_c^T (tcgen05, K = 64)  ->  Z += sum_j EXP[S_j]            (table of exp(fl32(s c)), fp64 sum)
//   pass B   S_c again                        ->  codes = min(rint(EXP[S_j] / (Z s_P)), Qp)  ->  P_c in shared memory
//            O += P_c V_c (tcgen05, accumulating in tensor memory across the chunks)
// Pass A needs the table's exact entries.  Pass B only needs the level they lead to, and finds it from 2^(s c2 + log2 r) on the
// special-function unit; blocks in which a score comes too close to a rounding boundary to be sure of take the table again.
// (Two ends of an interval as in the Eq. 4 core instead of |a - rint(a)| compared with a limit: an interval grows with a, and a
// clamp costs what it saves.  785 tokens x 12 heads, batch 16: 162.9 us against 162.2, rows that peak at one token 163.0 against
// 160.8, a step of 2e-5 172 against 161; 577 tokens 92.8 against 94.2.)
// So the lookups -- 2.8 passes of the shared-memory pipe per 32 scores, what bounded the kernel with two a score -- are halved.
// then O is requantized and stored.  S, the probabilities and P never reach HBM: the unfused sequence writes and
// re-reads 4 T^2 bytes per head (946 MB at 785 tokens, batch 32), which is what bounds it.  The table makes the
// two-pass form exact and cheap: exp(t_j) / sum_k exp(t_k) needs no running maximum and no rescaling of O, and Q K^T
// (a K = 64 contraction) costs next to nothing to repeat.  Arithmetic per score is that of attention_fused_kernel,
// so the codes are the same.
//
// One pipeline per CTA, steps in sequence (every thread passes the same barriers; an expired wait makes the whole CTA
// leave together), two CTAs per SM so that one's loads and MMAs run beside the other's softmax.  A step ends with one barrier
// of the CTA, behind which the control warp issues P V of this chunk and Q K^T of the next (of the other pass, of the next
// item) under one completion; the K behind that is requested at the same time, and V is awaited only in front of P V.  Items are numbered by query tile first,
// so that the last tile of every head, often nearly empty, fills the last round.  Byte-stored codes.
// 785 tokens x 12 heads, batch 16: 202 -> 160 us (with a wait and a barrier more per chunk, Q K^T issued behind them, 162).
#include "common.cuh"
#include "ptx.cuh"
#include "tile_ops.cuh"

namespace vitint {
namespace {

constexpr int AL_COMPUTE_WARPS = 8;     // two threads per query row, alternate 32-column blocks
constexpr int AL_THREADS = (AL_COMPUTE_WARPS + 1) * 32;
constexpr int AL_MAX_CHUNK = 192;       // S chunk (192 columns) + O (64 columns) = the CTA's 256 tensor-memory columns
constexpr uint32_t AL_O_COL = 192;

struct LongParams {
    int batch, heads, tokens, q_tiles, total_items;
    int chunk, n_chunks;          // keys per chunk (multiple of 32), chunks per row
    int smax;
    int part_bytes;               // bytes of one of the Q / K / V segments in a QKV row
    const float* table;
    float p_step, p_qp, c2;       // c2: the scores' scale in the exponent of two
    const float* alpha_o;
    const float* beta_o;
    uint8_t* out;
    int64_t out_pitch;
    int out_c;
    float out_qn, out_qp;
    uint32_t k_stride;            // bytes between the two K buffers
    uint32_t off_table, off_q, off_k, off_v, off_p, off_z, off_col;
};

struct LongBars {
    uint64_t q_full, k_full[2], v_full, s_full;
};

__global__ void __launch_bounds__(AL_THREADS, 2)
attention_long_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kv,
                      const __grid_constant__ LongParams P) {
    extern __shared__ uint8_t al_smem_raw[];
    __shared__ LongBars B;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t smem_base = (ptx::smem_addr(al_smem_raw) + 1023u) & ~1023u;
    uint8_t* const smem_gen = al_smem_raw + (smem_base - ptx::smem_addr(al_smem_raw));
    volatile int* abort_ptr = &abort_flag;
    const bool is_control = warp == AL_COMPUTE_WARPS;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        ptx::mbar_init(ptx::smem_addr(&B.q_full), 1);
        ptx::mbar_init(ptx::smem_addr(&B.k_full[0]), 1);
        ptx::mbar_init(ptx::smem_addr(&B.k_full[1]), 1);
        ptx::mbar_init(ptx::smem_addr(&B.v_full), 1);
        ptx::mbar_init(ptx::smem_addr(&B.s_full), 1);
        ptx::fence_mbar_init();
        ptx::fence_proxy_async_smem();
    }
    if (is_control) {
        ptx::tmem_alloc(ptx::smem_addr(&tmem_base_slot), 256);
        ptx::tmem_relinquish();
    }
    grid_dependency_wait();        // the table and the codes come from earlier kernels of the stream
    grid_dependency_launch();
    {
        fill_table_ring(reinterpret_cast<float*>(smem_gen + P.off_table), P.table, P.smax, threadIdx.x, AL_THREADS);
    }
    if (is_control && lane == 0) { ptx::prefetch_tensormap(&map_q); ptx::prefetch_tensormap(&map_kv); }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base_slot, 0);

    const int T = P.tokens, CH = P.chunk;
    const uint32_t q_bytes = 128u * 64u, kv_bytes = (uint32_t)CH * 64u;
    const uint32_t idesc_qk = ptx::idesc_i8(128, CH, 1, 1, 0);
    const uint32_t idesc_pv = ptx::idesc_i8(128, 64, 0, 1, 1);
    const uint64_t q_desc = ptx::smem_desc(smem_base + P.off_q, 16, 512, ptx::SWIZZLE_64B);
    const uint64_t k_desc[2] = {ptx::smem_desc(smem_base + P.off_k, 16, 512, ptx::SWIZZLE_64B),
                                ptx::smem_desc(smem_base + P.off_k + P.k_stride, 16, 512, ptx::SWIZZLE_64B)};
    const uint64_t v_desc = ptx::smem_desc(smem_base + P.off_v, 16, 512, ptx::SWIZZLE_64B);
    const int pv_steps = CH / 32, blocks = CH / 32;

    // compute-thread coordinates (the control warp carries them along unused)
    const int wq = warp & 3;                                     // tensor-memory lane quarter
    const int hf = (warp >> 2) & 1;                              // which of the row's two threads
    const int tid_c = warp * 32 + lane;                          // 0..255 for compute threads
    const int row = wq * 32 + lane;
    const uint32_t t_row = tmem + ((uint32_t)(wq * 32) << 16);
    const char* const ring = reinterpret_cast<const char*>(smem_gen + P.off_table);
    const uint32_t ring_mask = 8u * (uint32_t)P.smax - 4u, qp2 = (uint32_t)P.p_qp * 0x00010001u;
    const bool steep = P.p_step < 1.0f / 65000.0f;               // codes before the clamp might not fit 16 bits
    const f32x2 c2 = f2_dup(P.c2);
    double* const zx = reinterpret_cast<double*>(smem_gen + P.off_z);
    float* const colp = reinterpret_cast<float*>(smem_gen + P.off_col);
    const double inv_p_step = 1.0 / (double)P.p_step;
    uint8_t* const prow = smem_gen + P.off_p + row * 128;
    const int sw = row & 7;

    uint32_t n_q = 0, n_k = 0, n_v = 0, n_s = 0;                 // completed phases of each barrier (parity = count & 1; K alternates)
    uint32_t i_q = 0, i_k = 0, i_v = 0;                          // copies issued (control warp)
    bool ok = true, w = true;                                    // w: every wait of this thread has been granted
    const int per_tile = P.batch * P.heads;
    auto coords = [&](int item, int& b, int& h, int& qt) {
        qt = item / per_tile;
        const int bh = item - qt * per_tile;
        b = bh / P.heads;
        h = bh - b * P.heads;
    };
    // A step is one chunk of one pass over an item.
    struct Step { int item, pass, c; };
    auto step_after = [&](Step t) {
        if (++t.c == P.n_chunks) {
            t.c = 0;
            if (t.pass == 0) t.pass = 1;
            else { t.pass = 0; t.item += (int)gridDim.x; }
        }
        return t;
    };
    auto load_q = [&](int item) {
        int b, h, qt;
        coords(item, b, h, qt);
        if (ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx(ptx::smem_addr(&B.q_full), q_bytes);
            ptx::tma_load_3d(smem_base + P.off_q, &map_q, ptx::smem_addr(&B.q_full), h * 64, qt * 128, b);
        }
        ++i_q;
    };
    auto load_k = [&](Step t) {
        int b, h, qt;
        coords(t.item, b, h, qt);
        const uint32_t bar = ptx::smem_addr(&B.k_full[i_k & 1u]);
        if (ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx(bar, kv_bytes);
            ptx::tma_load_3d(smem_base + P.off_k + (i_k & 1u) * P.k_stride, &map_kv, bar, P.part_bytes + h * 64, t.c * CH, b);
        }
        ++i_k;
    };
    // Q K^T of step t into S, and the K of the step behind it (the other K buffer was read by the product before this one, which
    // has been awaited)
    auto issue_qk = [&](Step t) {
        if (t.pass == 0 && t.c == 0) { w = w && mbar_wait_warp(ptx::smem_addr(&B.q_full), n_q & 1u, abort_ptr); ++n_q; }
        w = w && mbar_wait_warp(ptx::smem_addr(&B.k_full[n_k & 1u]), (n_k >> 1) & 1u, abort_ptr);
        if (!w) return;
        ptx::tc_fence_after();
        const uint64_t kd = k_desc[n_k & 1u];
        if (ptx::elect_one()) {
            for (int k = 0; k < 2; ++k)
                ptx::mma_i8(tmem, q_desc + (uint64_t)(k * 2), kd + (uint64_t)(k * 2), idesc_qk, k);
        }
        __syncwarp();
        ++n_k;
        const Step next = step_after(t);
        if (next.item < P.total_items) load_k(next);
    };
    if (is_control && (int)blockIdx.x < P.total_items) {
        const Step first{(int)blockIdx.x, 0, 0};
        load_q(first.item);
        load_k(first);
        issue_qk(first);
        if (w && ptx::elect_one()) ptx::mma_commit(ptx::smem_addr(&B.s_full));
        __syncwarp();
    }
    w = w && mbar_wait(ptx::smem_addr(&B.s_full), 0u, abort_ptr);
    n_s = 1;
    for (int item = blockIdx.x; ok && item < P.total_items; item += gridDim.x) {
        int b, h, qt;
        coords(item, b, h, qt);
        double zp[4] = {0.0, 0.0, 0.0, 0.0};
        f32x2 rzh2 = f2_dup(0.0f), rzl2 = f2_dup(0.0f), l2 = f2_dup(0.0f);
        float limit = 0.0f, e_top = 0.0f;
        const bool warp_live = qt * 128 + wq * 32 < T;
        for (int pass = 0; ok && pass < 2; ++pass) {
            for (int c = 0; ok && c < P.n_chunks; ++c) {
                const int key0 = c * CH;
                w = __all_sync(0xffffffffu, w);
                if (is_control && w) {
                    if (pass) {
                        // (the V before it has been read: P V completed with the scores at hand)
                        if (ptx::elect_one()) {
                            ptx::mbar_arrive_expect_tx(ptx::smem_addr(&B.v_full), kv_bytes);
                            ptx::tma_load_3d(smem_base + P.off_v, &map_kv, ptx::smem_addr(&B.v_full), 2 * P.part_bytes + h * 64, key0, b);
                        }
                        ++i_v;
                        // Q has been read for the last time
                        if (c + 1 == P.n_chunks && item + (int)gridDim.x < P.total_items) load_q(item + (int)gridDim.x);
                    }
                }
                ptx::tc_fence_after();
                if (!is_control && w && warp_live) {
                    if (pass == 0) {
                        // ---- pass A: row sum of the table entries ------------------------------------------
#pragma unroll 1
                        for (int blk = hf; blk < blocks; blk += 2) {
                            const int n_valid = T - (key0 + blk * 32);                  // columns of this block that are tokens
                            if (n_valid <= 0) break;
                            uint32_t v0[16], v1[16];
                            ptx::tmem_ld16(t_row + (uint32_t)(blk * 32), v0);
                            ptx::tmem_ld_wait();
                            ptx::tmem_ld16(t_row + (uint32_t)(blk * 32 + 16), v1);
                            if (n_valid >= 32) {
                                exp_lookup<16, false, false>(v0, ring, ring_mask, 0, 16, zp);
                                ptx::tmem_ld_wait();
                                exp_lookup<16, false, false>(v1, ring, ring_mask, 0, 16, zp);
                            } else {
                                exp_lookup<16, false, true>(v0, ring, ring_mask, 0, n_valid, zp);
                                ptx::tmem_ld_wait();
                                if (n_valid > 16) exp_lookup<16, false, true>(v1, ring, ring_mask, 0, n_valid - 16, zp);
                            }
                        }
                    } else {
                        // ---- pass B: codes of this chunk into the P tile -----------------------------------
#pragma unroll 1
                        for (int p16 = hf; p16 < 2 * blocks; p16 += 2) {               // the row's threads take 16 columns in turn
                            const int n_valid = T - (key0 + p16 * 16);
                            uint32_t wd[4] = {0u, 0u, 0u, 0u};
                            if (n_valid > 0) {
                                uint32_t v[16];
                                ptx::tmem_ld16(t_row + (uint32_t)(p16 * 16), v);
                                ptx::tmem_ld_wait();
                                bool sure = !steep && n_valid >= 16;
                                if (sure) sure = quantize_scores<16>(v, c2, l2, P.p_qp, limit, wd);
                                if (!__all_sync(0xffffffffu, sure)) {
                                    double unused[4] = {0.0, 0.0, 0.0, 0.0};
                                    exp_lookup<16, false, true>(v, ring, ring_mask, 0, n_valid, unused);
                                    if (steep) {
#pragma unroll
                                        for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(fminf(__uint_as_float(v[i]), e_top));
                                    }
                                    quantize_entries<16>(v, rzh2, rzl2, qp2, wd);
                                }
                            }
                            *reinterpret_cast<uint4*>(prow + (p16 >> 3) * 16384 + (((p16 & 7) ^ sw) << 4)) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                        }
                        ptx::fence_proxy_async_smem();
                    }
                }
                const bool last = c + 1 == P.n_chunks;
                if (pass == 0 && last && !is_control) {
                    zx[hf * 128 + row] = (zp[0] + zp[1]) + (zp[2] + zp[3]);
                    // the head's output parameters: at least two chunks, so a barrier lies behind the last item's use of them
                    if (tid_c < 64) colp[tid_c] = __ldg(P.alpha_o + h * 64 + tid_c);
                    else if (tid_c < 128) colp[tid_c] = P.beta_o ? __ldg(P.beta_o + h * 64 + (tid_c - 64)) : 0.0f;
                }
                ptx::tc_fence_before();
                if (!__syncthreads_and(w ? 1 : 0)) { ok = false; break; }        // S has been read; the P tile is complete
                if (is_control) {
                    if (pass == 1) {
                        // ---- O += P_c V_c ----------------------------------------------------------------------
                        w = mbar_wait_warp(ptx::smem_addr(&B.v_full), n_v & 1u, abort_ptr);
                        ++n_v;
                        if (w) {
                            ptx::tc_fence_after();
                            if (ptx::elect_one()) {
                                for (int ks = 0; ks < pv_steps; ++ks) {
                                    const uint64_t p_desc = ptx::smem_desc(smem_base + P.off_p + (uint32_t)(ks >> 2) * 16384u, 16, 1024,
                                                                           ptx::SWIZZLE_128B) + (uint64_t)((ks & 3) * 2);
                                    ptx::mma_i8(tmem + AL_O_COL, p_desc, v_desc + (uint64_t)(ks * 128), idesc_pv, (c > 0 || ks > 0) ? 1 : 0);
                                }
                            }
                            __syncwarp();
                        }
                    }
                    const Step next = step_after(Step{item, pass, c});
                    if (next.item < P.total_items && w) issue_qk(next);
                    if (w && ptx::elect_one()) ptx::mma_commit(ptx::smem_addr(&B.s_full));
                    __syncwarp();
                }
                if (pass == 0 && last && !is_control) {
                    // the row's two threads add their partial sums; r = 1 / (Z s_P) as a two-float number
                    const double z = zx[row] + zx[128 + row];
                    const double rz = warp_live ? inv_p_step / z : 0.0;
                    const float rzh = (float)rz;
                    rzh2 = f2_dup(rzh);
                    rzl2 = f2_dup((float)(rz - (double)rzh));
                    e_top = 60000.0f / rzh;                             // (steep only) far above Qp, below 2^16
                    // Pass B's exponent is s c2 + l.  Where the code is not 0 the exponent lies in [-1, 8], so |s c2| <= |l| + 8,
                    // and the roundings of c2, of l and of the FMA and the error of log2f leave at most (4 |l| + 40) 2^-24 in it
                    // and ln 2 times that, plus exp2's 2^-22, relative in the argument.
                    const float l = log2f(rzh);
                    l2 = f2_dup(l);
                    limit = 0.5f - (P.p_qp + 1.0f) * 1.25f * ((4.0f * fabsf(l) + 40.0f) * 4.1316e-8f + 2.4e-7f);
                }
                // the next step's scores (the last step of all: P V alone)
                w = w && mbar_wait(ptx::smem_addr(&B.s_full), n_s & 1u, abort_ptr);
                ++n_s;
            }
        }
        if (!ok) break;
        // ---- requantize O and store -------------------------------------------------------------------------
        ptx::tc_fence_after();
        if (!is_control && __all_sync(0xffffffffu, w)) {
            const int token = qt * 128 + row;
            uint32_t v[32], ow[8];
            ptx::tmem_ld32(t_row + AL_O_COL + (uint32_t)(hf * 32), v);
            ptx::tmem_ld_wait();
            // (once an item, so the conversion instruction: 8-bit P over more than 2056 tokens can take |O| past 2^22)
            requantize_row<false, 32>(v, 0, colp + hf * 32, colp + 64 + hf * 32, P.out_qn, P.out_qp, ow);
            if (token < T) {
                store_row(P.out + ((long long)b * T + token) * P.out_pitch + (long long)h * (8 * P.out_c) + hf * (4 * P.out_c), ow, P.out_c);
                if (h == P.heads - 1 && hf == 1) {
                    uint8_t* const orow = P.out + ((long long)b * T + token) * P.out_pitch;
                    for (long long off = (long long)P.heads * (8 * P.out_c); off + 4 <= P.out_pitch; off += 4)
                        *reinterpret_cast<uint32_t*>(orow + off) = 0u;
                }
            }
        }
        ptx::tc_fence_before();                                         // (O is written again a whole pass of barriers later)
    }
    ok = ok && w;
    // copies still in flight when the CTA gives up are given a bounded chance to land
    if (!ok && is_control) {
        auto drain = [&](uint64_t* bar, uint32_t issued) {               // the last phase of a barrier that was armed `issued` times
            for (int spin = 0; spin < (1 << 20) && issued > 0 && !ptx::mbar_try_wait(ptx::smem_addr(bar), (issued - 1u) & 1u); ++spin) {}
        };
        drain(&B.q_full, i_q);
        drain(&B.k_full[0], (i_k + 1u) >> 1);
        drain(&B.k_full[1], i_k >> 1);
        drain(&B.v_full, i_v);
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (is_control) {
        ptx::tc_fence_after();
        __syncwarp();
        ptx::tmem_dealloc(tmem_base_slot, 256);
    }
}

inline uint32_t al_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

}  // namespace

// Launcher shared with attention_core_launch: byte-stored codes, more than 256 tokens, table already in `table`.
int attention_long_launch(const vitint_codes* qkv, int batch, int heads, int tokens, int smax, const float* table, float cs, float p_step,
                          float p_qp, const float* alpha_o, const float* beta_o, const vitint_codes* o_out, cudaStream_t st) {
    const int64_t D = (int64_t)heads * 64;
    LongParams P{};
    P.batch = batch; P.heads = heads; P.tokens = tokens;
    P.q_tiles = (tokens + 127) / 128;
    const long long items = (long long)batch * heads * P.q_tiles;
    if (items > 0x7fffffffll) return VITINT_ERR_UNSUPPORTED;
    P.total_items = (int)items;
    P.n_chunks = (tokens + AL_MAX_CHUNK - 1) / AL_MAX_CHUNK;
    P.chunk = ((tokens + P.n_chunks - 1) / P.n_chunks + 31) / 32 * 32;          // <= 192, a multiple of 32
    P.smax = smax;
    P.part_bytes = (int)D;
    P.table = table;
    P.p_step = p_step; P.p_qp = p_qp;
    P.c2 = (float)((double)cs * 1.4426950408889634);
    P.alpha_o = alpha_o; P.beta_o = beta_o;
    P.out_c = codes_container(o_out);
    int qn, qp;
    code_range(o_out->bits, o_out->is_signed, &qn, &qp);
    P.out_qn = (float)qn; P.out_qp = (float)qp;
    P.out = (uint8_t*)o_out->data; P.out_pitch = o_out->pitch_bytes;
    uint32_t o = 0;
    P.off_table = o; o += al_up((uint32_t)(2 * smax) * 4u, 1024);
    P.off_q = o; o += 128 * 64;
    P.k_stride = al_up((uint32_t)P.chunk * 64, 1024);
    P.off_k = o; o += 2 * P.k_stride;
    P.off_v = o; o += al_up((uint32_t)P.chunk * 64, 1024);
    P.off_p = o; o += (uint32_t)((P.chunk + 127) / 128) * 16384u;
    P.off_z = o; o += 2 * 128 * 8;
    P.off_col = o; o += 512;
    const size_t smem = (size_t)o + 1024;
    if (smem > 113 * 1024) return VITINT_ERR_UNSUPPORTED;                       // two CTAs per SM

    CUtensorMap map_q, map_kv;
    {
        EncodeTiledFn fn = encode_fn();
        if (!fn) return VITINT_ERR_CUDA;
        cuuint64_t dims[3] = {(cuuint64_t)codes_row_bytes(qkv, 3 * D), (cuuint64_t)tokens, (cuuint64_t)batch};
        cuuint64_t strides[2] = {(cuuint64_t)qkv->pitch_bytes, (cuuint64_t)qkv->pitch_bytes * tokens};
        cuuint32_t estr[3] = {1, 1, 1};
        cuuint32_t box_q[3] = {64, 128, 1}, box_kv[3] = {64, (cuuint32_t)P.chunk, 1};
        if (fn(&map_q, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, qkv->data, dims, strides, box_q, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
            fn(&map_kv, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, qkv->data, dims, strides, box_kv, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return VITINT_ERR_CUDA;
    }
    int grid = 2 * sm_count();
    if (grid > P.total_items) grid = P.total_items;
    const int dev = current_device();
    if (dev < 0) return VITINT_ERR_CUDA;
    static bool attr_set_dev[MAX_DEVICES] = {};
    if (!attr_set_dev[dev]) {
        if (cudaFuncSetAttribute(attention_long_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024) != cudaSuccess)
            return VITINT_ERR_CUDA;
        attr_set_dev[dev] = true;
    }
    launch_kernel(attention_long_kernel, dim3(grid), dim3(AL_THREADS), smem, st, map_q, map_kv, P);
    return cuda_status(cudaGetLastError());
}

}  // namespace vitint

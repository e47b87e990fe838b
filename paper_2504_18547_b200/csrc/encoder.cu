// A stack of encoder layers as one host call (Fig. 1(b) layer after layer), launch by launch or as a recorded graph.
//
// Why a graph: a launch costs the host about 4 us (tensor maps of a GEMM 2 us more), while at one image a layer's seven
// kernels run for 3 to 9 us each, so launches one by one are what a small batch waits for.  A graph launch costs the host
// little per kernel; x and out of a call enter through the parameters of the first layer's LayerNorm and projection and the
// last layer's fc2, which are rewritten before each launch.
#include <exception>
#include <memory>
#include <mutex>

#include "common.cuh"

namespace vitint {

namespace {

enum Stage { ST_LN1, ST_QKV, ST_ATTENTION, ST_PROJ, ST_LN2, ST_FC1, ST_FC2, NUM_STAGES };

// What the C++ library throws (no host memory, a lock that fails) ends here as a status: a plan's functions are called from C.
template <typename F>
int no_exceptions(F&& f) {
    try {
        return f();
    } catch (const std::exception&) {
        return VITINT_ERR_CUDA;
    }
}

// A plan is made and destroyed in calls that a stream capture elsewhere in the process (or on this thread) would otherwise count
// against itself: they touch no stream, so the thread leaves the capture's restrictions for their time.
struct OutsideCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

struct RecorderScope {
    explicit RecorderScope(LaunchRecorder* r) { t_recorder = r; }
    ~RecorderScope() { t_recorder = nullptr; }
};

// tables_ready: the table of the bounded softmax has been filled (by vitint_encoder_plan_create); otherwise the softmax fills it.
int attention_stage(const vitint_encoder_layer_desc& L, bool tables_ready, void* stream) {
    const int64_t D = (int64_t)L.heads * 64;
    if (L.attention == VITINT_ATTN_EXP_CORE)
        return vitint_attention_core_prepared(&L.qkv, L.batch, L.heads, L.tokens, L.q_step, L.k_step, L.p_step, L.bits, L.alpha_o,
                                              nullptr, &L.o, L.table, L.table_bytes, stream);
    if (L.attention == VITINT_ATTN_SHIFT_CORE)
        return vitint_attention_core_shift(&L.qkv, L.batch, L.heads, L.tokens, L.q_step, L.k_step, L.p_step, L.bits, L.alpha_o,
                                           nullptr, &L.o, L.table, L.table_bytes, 1, stream);
    if (L.attention == VITINT_ATTN_EXP_CORE_ANY)
        return attention_core_general(&L.qkv, L.batch, L.heads, L.tokens, L.q_step, L.k_step, L.p_step, L.bits, L.alpha_o, nullptr, &L.o,
                                      stream);
    const int c = container_bits(L.bits);
    vitint_slabs q{L.qkv.data, L.qkv.pitch_bytes, L.qkv.pitch_bytes * L.tokens, 64 * c / 8, L.bits, 1};
    vitint_slabs k = q, v = q;
    k.data = (const uint8_t*)L.qkv.data + D * c / 8;
    v.data = (const uint8_t*)L.qkv.data + 2 * D * c / 8;
    const int64_t rows = (int64_t)L.batch * L.heads * L.tokens;
    if (int rc = vitint_qk(&q, &k, L.batch, L.heads, L.tokens, L.scores, L.ld_scores, stream)) return rc;
    int rc;
    if (L.attention == VITINT_ATTN_SHIFT)
        rc = vitint_softmax_shift_quantize(L.scores, rows, L.tokens, L.ld_scores, L.c, L.p_step, &L.p, stream);
    else if (L.attention == VITINT_ATTN_EXP_BOUNDED)
        rc = vitint_softmax_quantize_bounded(L.scores, rows, L.tokens, L.ld_scores, L.c, L.p_step, L.score_bound, &L.p, nullptr, 0,
                                             L.table, L.table_bytes, tables_ready ? 1 : 0, stream);
    else
        rc = vitint_softmax_quantize(L.scores, rows, L.tokens, L.ld_scores, L.c, L.p_step, &L.p, nullptr, 0, stream);
    if (rc) return rc;
    vitint_epilogue e{};
    e.mode = VITINT_EPI_REQUANT; e.alpha = L.alpha_o; e.out_bits = L.o.bits; e.out_signed = 1; e.out_container_bits = L.o.container_bits;
    return vitint_pv(&L.p, &v, L.batch, L.heads, L.tokens, L.p_step, L.v_step, &e, L.o.data, L.o.pitch_bytes, stream);
}

int run_stage(const vitint_encoder_layer_desc& L, int stage, const float* x, float* out, bool tables_ready, void* stream) {
    const int64_t D = (int64_t)L.heads * 64, M = (int64_t)L.batch * L.tokens;
    vitint_epilogue e{};
    switch (stage) {
        case ST_LN1:
        case ST_LN2: {
            const bool first = stage == ST_LN1;
            const float* in = first ? x : L.h;
            const vitint_codes* codes = first ? &L.x1 : &L.x2;
            if (L.compare_layernorm)
                return vitint_layernorm_compare_quantize(in, M, D, D, first ? L.ln1_refs : L.ln2_refs, first ? L.ln1_flip : L.ln2_flip,
                                                         L.n_eps, codes, L.ln_stats, stream);
            return vitint_layernorm_quantize(in, M, D, D, first ? L.ln1_gamma : L.ln2_gamma, first ? L.ln1_beta : L.ln2_beta, L.eps,
                                             L.ln_step, codes, nullptr, 0, stream);
        }
        case ST_QKV:
            e.mode = VITINT_EPI_REQUANT; e.alpha = L.alpha_qkv; e.beta = L.beta_qkv;
            e.out_bits = L.qkv.bits; e.out_signed = 1; e.out_container_bits = L.qkv.container_bits;
            return vitint_linear(&L.x1, L.ln_step, &L.w_qkv, nullptr, nullptr, &e, L.qkv.data, L.qkv.pitch_bytes, stream);
        case ST_ATTENTION:
            return attention_stage(L, tables_ready, stream);
        case ST_PROJ:
            e.mode = VITINT_EPI_DEQUANT_F32; e.residual = x; e.ld_res = D;
            return vitint_linear(&L.o, L.o_step, &L.w_proj, L.proj_step, L.proj_bias, &e, L.h, D, stream);
        case ST_FC1:
            e.mode = VITINT_EPI_REQUANT; e.act = 1; e.inv_out_step = L.inv_g_step;
            e.out_bits = L.g.bits; e.out_signed = 0; e.out_container_bits = L.g.container_bits;
            return vitint_linear(&L.x2, L.ln_step, &L.w_fc1, L.fc1_step, L.fc1_bias, &e, L.g.data, L.g.pitch_bytes, stream);
        default:
            e.mode = VITINT_EPI_DEQUANT_F32; e.residual = L.h; e.ld_res = D;
            return vitint_linear(&L.g, L.g_step, &L.w_fc2, L.fc2_step, L.fc2_bias, &e, out, D, stream);
    }
}

// stage_end, when given, receives the number of launches recorded up to the end of every stage.
int run_stack(const vitint_encoder_layer_desc* layers, int n, float* const buf[2], const float* x, float* out, bool tables_ready,
              void* stream, std::vector<size_t>* stage_end = nullptr) {
    const float* cur = x;
    for (int i = 0; i < n; ++i) {
        float* const dst = i + 1 == n ? out : buf[i & 1];
        for (int s = 0; s < NUM_STAGES; ++s) {
            if (int rc = run_stage(layers[i], s, cur, dst, tables_ready, stream)) return rc;
            if (stage_end) stage_end->push_back(t_recorder->next);
        }
        cur = dst;
    }
    return VITINT_OK;
}

// What no stage checks by itself: that a layer's matrices have the rows the stages around them write or read, and the table that
// vitint_encoder_plan_create fills in front of any stage.
int check_stack(const vitint_encoder_layer_desc* layers, int n, float* const buf[2]) {
    if (!layers || n <= 0 || (n > 1 && (!buf || !buf[0] || (n > 2 && !buf[1])))) return VITINT_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i) {
        const vitint_encoder_layer_desc& L = layers[i];
        if (L.batch <= 0 || L.tokens <= 0 || L.heads <= 0 || !L.h || L.attention < VITINT_ATTN_EXP_CORE || L.attention > VITINT_ATTN_EXP_CORE_ANY)
            return VITINT_ERR_INVALID_ARG;
        const int64_t D = (int64_t)L.heads * 64, M = (int64_t)L.batch * L.tokens;
        if (L.qkv.rows != M || L.o.rows != M || L.g.rows != M || L.w_qkv.rows != 3 * D || L.w_proj.rows != D || L.w_fc1.rows != L.g.cols ||
            L.w_fc2.rows != D)
            return VITINT_ERR_INVALID_ARG;
        if (L.attention == VITINT_ATTN_EXP_BOUNDED) {
            const size_t need = vitint_softmax_table_workspace_bytes(L.score_bound);
            if (need == 0) return L.score_bound <= 0 ? VITINT_ERR_INVALID_ARG : VITINT_ERR_UNSUPPORTED;
            if (!L.table || (reinterpret_cast<uintptr_t>(L.table) & 255u) || L.table_bytes < need) return VITINT_ERR_WORKSPACE;
        }
    }
    return VITINT_OK;
}

}  // namespace
}  // namespace vitint

using namespace vitint;

struct vitint_encoder_plan {
    std::vector<vitint_encoder_layer_desc> layers;
    float* buf[2];
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<cudaGraphNode_t> nodes;
    std::vector<size_t> stage_end;            // launches up to the end of layer i, stage s: [i * NUM_STAGES + s]
    std::mutex lock;                          // the instance's parameters are rewritten before each launch
    ~vitint_encoder_plan() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
    int update(int layer, int stage, const float* x, float* out) {
        const size_t at = (size_t)layer * NUM_STAGES + (size_t)stage, first = at ? stage_end[at - 1] : 0;
        LaunchRecorder r;
        r.exec = exec; r.nodes = &nodes; r.next = first;
        RecorderScope scope(&r);
        if (int rc = run_stage(layers[(size_t)layer], stage, x, out, true, nullptr)) return rc;
        return r.error == cudaSuccess && r.next == stage_end[at] ? VITINT_OK : VITINT_ERR_CUDA;
    }
};

extern "C" int vitint_encoder_forward(const vitint_encoder_layer_desc* layers, int32_t n_layers, float* const buf[2], const float* x,
                                      float* out, void* stream) {
    if (int rc = check_stack(layers, n_layers, buf)) return rc;
    if (!x || !out) return VITINT_ERR_INVALID_ARG;
    return run_stack(layers, n_layers, buf, x, out, false, stream);
}

extern "C" int vitint_encoder_plan_create(const vitint_encoder_layer_desc* layers, int32_t n_layers, float* const buf[2], void* stream,
                                          vitint_encoder_plan** plan) {
    if (!plan) return VITINT_ERR_INVALID_ARG;
    if (int rc = check_stack(layers, n_layers, buf)) return rc;
    *plan = nullptr;
    return no_exceptions([&]() -> int {
        OutsideCapture outside;
        std::unique_ptr<vitint_encoder_plan> p(new vitint_encoder_plan);
        p->layers.assign(layers, layers + n_layers);
        p->buf[0] = buf ? buf[0] : nullptr;
        p->buf[1] = buf ? buf[1] : nullptr;
        int rc = VITINT_OK;
        if (rc == VITINT_OK && cudaGraphCreate(&p->graph, 0) != cudaSuccess) rc = VITINT_ERR_CUDA;
        if (rc == VITINT_OK) {
            // recorded with the intermediate buffer in place of x and out; every run sets its own
            LaunchRecorder r;
            r.graph = p->graph; r.nodes = &p->nodes;
            RecorderScope scope(&r);
            float* const io = p->layers[0].h;
            rc = run_stack(p->layers.data(), n_layers, p->buf, io, io, true, nullptr, &p->stage_end);
            if (rc == VITINT_OK && r.error != cudaSuccess) rc = VITINT_ERR_CUDA;
        }
        // (behind the stages' own checks, which recording has run)
        for (const vitint_encoder_layer_desc& L : p->layers) {
            if (rc == VITINT_OK && L.attention == VITINT_ATTN_EXP_BOUNDED)
                rc = softmax_bounded_table(L.c, L.score_bound, L.table, L.table_bytes, (cudaStream_t)stream);
        }
        if (rc == VITINT_OK && cudaGraphInstantiate(&p->exec, p->graph, 0) != cudaSuccess) rc = VITINT_ERR_CUDA;
        if (rc == VITINT_OK) *plan = p.release();
        return rc;
    });
}

extern "C" int vitint_encoder_plan_run(vitint_encoder_plan* plan, const float* x, float* out, void* stream) {
    if (!plan || !x || !out) return VITINT_ERR_INVALID_ARG;
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing((cudaStream_t)stream, &capturing) != cudaSuccess) return VITINT_ERR_CUDA;
    const int n = (int)plan->layers.size();
    if (capturing != cudaStreamCaptureStatusNone) return run_stack(plan->layers.data(), n, plan->buf, x, out, true, stream);
    return no_exceptions([&]() -> int {
        std::lock_guard<std::mutex> guard(plan->lock);
        if (int rc = plan->update(0, ST_LN1, x, nullptr)) return rc;
        if (int rc = plan->update(0, ST_PROJ, x, nullptr)) return rc;
        if (int rc = plan->update(n - 1, ST_FC2, nullptr, out)) return rc;
        return cuda_status(cudaGraphLaunch(plan->exec, (cudaStream_t)stream));
    });
}

extern "C" void vitint_encoder_plan_destroy(vitint_encoder_plan* plan) {
    OutsideCapture outside;
    delete plan;
}

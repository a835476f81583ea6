// C-ABI entry points of the hyq library: argument checks on the host, then kernel launches.
#include <cmath>

#include "attn_common.cuh"
#include "quantize.cuh"
#include "select_common.cuh"

namespace hyq {
size_t attn_simt_workspace_bytes(const hyq_attn_args& a);
int launch_attn_simt(const hyq_attn_args& a, float alpha, cudaStream_t st);
int tc_restarts(unsigned long long* count, bool reset);
namespace tcbt {
int tc_restarts(unsigned long long* count, bool reset);
}
}  // namespace hyq

namespace hyq {
static TcTestHooks g_tc_hooks = {0, -1};
TcTestHooks tc_test_hooks() { return g_tc_hooks; }
}  // namespace hyq

using namespace hyq;

extern "C" {

const char* hyq_status_string(int status) {
    switch (status) {
        case HYQ_OK: return "ok";
        case HYQ_ERR_INVALID_ARG: return "invalid argument";
        case HYQ_ERR_UNSUPPORTED: return "unsupported shape or format";
        case HYQ_ERR_WORKSPACE: return "workspace too small";
        case HYQ_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
        case HYQ_ERR_CUDA: return "CUDA call failed";
        case HYQ_ERR_TIMEOUT: return "bounded device wait expired";
        default: return "unknown status";
    }
}

int hyq_version(void) { return 2; }   // 2: decode side, column-mass selector, block sizes

int hyq_test_set_attention_hooks(long long wait_limit_clocks, int drop_load_position) {
    if (wait_limit_clocks < 0 || drop_load_position < -1) return HYQ_ERR_INVALID_ARG;
    g_tc_hooks.wait_limit = wait_limit_clocks;
    g_tc_hooks.drop_load = drop_load_position;
    return HYQ_OK;
}

int hyq_test_read_attention_restarts(unsigned long long* count_out, int reset) {
    if (!count_out) return HYQ_ERR_INVALID_ARG;
    unsigned long long a = 0ull, b = 0ull;
    if (tc_restarts(&a, reset != 0) != HYQ_OK || tcbt::tc_restarts(&b, reset != 0) != HYQ_OK) return HYQ_ERR_CUDA;
    *count_out = a + b;
    return HYQ_OK;
}

int hyq_paper_k(int Lk, int window, double ratio) {
    const long P = (Lk - window > 0) ? (long)Lk - window : 0;
    if (P == 0) return 0;
    long k = (long)std::ceil((double)P * ratio);
    if (k < 1) k = 1;
    if (k > P) k = P;
    return (int)k;
}

static int check_select(const void* q, const void* k_, int B, int Hq, int Hkv, int Lq, int Lk, int D, int window,
                        int n_tail, int k) {
    if (B <= 0 || Hq <= 0 || Hkv <= 0 || Lq <= 0 || Lk <= 0 || window < 0 || k < 0 || n_tail < 0) return HYQ_ERR_INVALID_ARG;
    if (Hq % Hkv) return HYQ_ERR_INVALID_ARG;
    if (D != HYQ_D) return HYQ_ERR_UNSUPPORTED;
    const long P = (Lk - window > 0) ? (long)Lk - window : 0;
    if (P == 0 || k == 0) return HYQ_OK;
    if (k > P || n_tail > Lq) return HYQ_ERR_INVALID_ARG;
    if (n_tail == 0 && window == 0) return HYQ_ERR_INVALID_ARG;    // mean of zero rows
    (void)q; (void)k_;
    return HYQ_OK;
}

int hyq_select_vertical_workspace(int B, int Hq, int Hkv, int Lq, int Lk, int D, int window, int k, size_t* bytes) {
    if (!bytes) return HYQ_ERR_INVALID_ARG;
    const int rc = check_select(nullptr, nullptr, B, Hq, Hkv, Lq, Lk, D, window, 1, k);
    if (rc != HYQ_OK) return rc;
    *bytes = select_workspace_bytes(B, Hq, Lk, window);
    return HYQ_OK;
}

int hyq_select_vertical(const void* q, const void* k_, int B, int Hq, int Hkv, int Lq, int Lk, int D, int window,
                        int n_tail, int k, int32_t* idx_out, void* workspace, size_t workspace_bytes, void* stream) {
    const int rc = check_select(q, k_, B, Hq, Hkv, Lq, Lk, D, window, n_tail, k);
    if (rc != HYQ_OK) return rc;
    const long P = (Lk - window > 0) ? (long)Lk - window : 0;
    if (P == 0 || k == 0) return HYQ_OK;
    if (!q || !k_ || !idx_out || !workspace) return HYQ_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k_) || !aligned16(workspace) || (reinterpret_cast<uintptr_t>(idx_out) & 3u))
        return HYQ_ERR_ALIGNMENT;
    if (workspace_bytes < select_workspace_bytes(B, Hq, Lk, window)) return HYQ_ERR_WORKSPACE;
    return launch_select(q, k_, B, Hq, Hkv, Lq, Lk, window, n_tail, k, idx_out, workspace, static_cast<cudaStream_t>(stream));
}

int hyq_select_vertical_static(const void* q, const void* k_, int B, int Hq, int Hkv, int Lq, int Lk, int D, int window,
                               int n_tail, int k, int32_t* idx_out, void* stream) {
    const int rc = check_select(q, k_, B, Hq, Hkv, Lq, Lk, D, window, n_tail, k);
    if (rc != HYQ_OK) return rc;
    const long P = (Lk - window > 0) ? (long)Lk - window : 0;
    if (P == 0 || k == 0) return HYQ_OK;
    if (!q || !k_ || !idx_out) return HYQ_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k_) || (reinterpret_cast<uintptr_t>(idx_out) & 3u)) return HYQ_ERR_ALIGNMENT;
    return launch_select_static(q, k_, B, Hq, Hkv, Lq, Lk, window, n_tail, k, idx_out, static_cast<cudaStream_t>(stream));
}

static int check_select_mass(int B, int Hq, int Hkv, int Lq, int Lk, int D, int window, int n_queries, int k, int* n_eff) {
    if (n_queries < 0) return HYQ_ERR_INVALID_ARG;
    const int rc = check_select(nullptr, nullptr, B, Hq, Hkv, Lq, Lk, D, window, n_queries, k);
    if (rc != HYQ_OK) return rc;
    const int tail = window < Lq ? window : Lq;
    *n_eff = n_queries ? n_queries : tail;
    const long P = (Lk - window > 0) ? (long)Lk - window : 0;
    if (P == 0 || k == 0) return HYQ_OK;
    if (Lq > Lk || *n_eff > tail || *n_eff <= 0) return HYQ_ERR_INVALID_ARG;
    return HYQ_OK;
}

int hyq_select_vertical_mass_workspace(int B, int Hq, int Hkv, int Lq, int Lk, int D, int window, int n_queries, int k,
                                       size_t* bytes) {
    if (!bytes) return HYQ_ERR_INVALID_ARG;
    int nT = 0;
    const int rc = check_select_mass(B, Hq, Hkv, Lq, Lk, D, window, n_queries, k, &nT);
    if (rc != HYQ_OK) return rc;
    *bytes = select_mass_query_bytes(B, Hq, Lk, window, nT);
    return HYQ_OK;
}

int hyq_select_vertical_mass(const void* q, const void* k_, int B, int Hq, int Hkv, int Lq, int Lk, int D, int window,
                             int n_queries, int k, float softmax_scale, int32_t* idx_out, void* workspace,
                             size_t workspace_bytes, void* stream) {
    int nT = 0;
    const int rc = check_select_mass(B, Hq, Hkv, Lq, Lk, D, window, n_queries, k, &nT);
    if (rc != HYQ_OK) return rc;
    const long P = (Lk - window > 0) ? (long)Lk - window : 0;
    if (P == 0 || k == 0) return HYQ_OK;
    if (!q || !k_ || !idx_out || !workspace) return HYQ_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k_) || !aligned16(workspace) || (reinterpret_cast<uintptr_t>(idx_out) & 3u))
        return HYQ_ERR_ALIGNMENT;
    if (workspace_bytes < select_mass_workspace_bytes(B, Hq, Lk, window, nT)) return HYQ_ERR_WORKSPACE;
    const double alpha = softmax_scale != 0.0f ? (double)softmax_scale : 1.0 / std::sqrt((double)D);
    return launch_select_mass(q, k_, B, Hq, Hkv, Lq, Lk, window, nT, k, alpha, idx_out, workspace,
                              static_cast<cudaStream_t>(stream));
}

int hyq_quantize_blocks(const void* x, int B, int H, int L, int D, int block_tokens, int format, void* codes_out,
                        float* scales_out, void* stream) {
    if (B <= 0 || H <= 0 || L <= 0) return HYQ_ERR_INVALID_ARG;
    if (!x || !codes_out || !scales_out) return HYQ_ERR_INVALID_ARG;
    if (D != HYQ_D || !block_tokens_ok(block_tokens)) return HYQ_ERR_UNSUPPORTED;
    if (format != HYQ_FMT_INT8 && format != HYQ_FMT_FP8_E4M3 && format != HYQ_FMT_INT4) return HYQ_ERR_UNSUPPORTED;
    if (!aligned16(x) || !aligned16(codes_out) || (reinterpret_cast<uintptr_t>(scales_out) & 3u)) return HYQ_ERR_ALIGNMENT;
    return launch_quantize(x, (long)B * H, L, block_tokens, format, codes_out, scales_out, static_cast<cudaStream_t>(stream));
}

static int check_attn(const hyq_attn_args* a, bool need_pointers) {
    if (!a || a->struct_size != sizeof(hyq_attn_args)) return HYQ_ERR_INVALID_ARG;
    if (a->B <= 0 || a->Hq <= 0 || a->Hkv <= 0 || a->L <= 0 || a->window < 0 || a->k < 0) return HYQ_ERR_INVALID_ARG;
    if (a->Hq % a->Hkv || a->k > a->L || a->Lq < 0 || a->Lq > a->L) return HYQ_ERR_INVALID_ARG;
    if (a->window_mode != HYQ_WINDOW_SLIDING && a->window_mode != HYQ_WINDOW_FIXED_TAIL) return HYQ_ERR_INVALID_ARG;
    if (a->out_dtype != 0 && a->out_dtype != 1) return HYQ_ERR_INVALID_ARG;
    if (a->impl < HYQ_IMPL_AUTO || a->impl > HYQ_IMPL_SIMT) return HYQ_ERR_INVALID_ARG;
    if (a->D != HYQ_D || !block_tokens_ok(a->block_tokens)) return HYQ_ERR_UNSUPPORTED;
    const bool int8 = a->q_format == HYQ_FMT_INT8 && a->k_format == HYQ_FMT_INT8 && a->v_format == HYQ_FMT_INT8;
    const bool int4 = a->q_format == HYQ_FMT_INT4 && a->k_format == HYQ_FMT_INT4 && a->v_format == HYQ_FMT_FP8_E4M3;
    const bool fp8 = a->q_format == HYQ_FMT_FP8_E4M3 && a->k_format == HYQ_FMT_FP8_E4M3 && a->v_format == HYQ_FMT_FP8_E4M3;
    if (!int8 && !int4 && !fp8) return HYQ_ERR_UNSUPPORTED;
    if (!need_pointers) return HYQ_OK;
    const void* ptrs[] = {a->q, a->k_, a->v, a->q_codes, a->k_codes, a->v_codes, a->q_scales, a->k_scales, a->v_scales, a->out};
    for (const void* p : ptrs)
        if (!p) return HYQ_ERR_INVALID_ARG;
    if (a->k > 0 && !a->vl_idx) return HYQ_ERR_INVALID_ARG;
    const void* al[] = {a->q, a->k_, a->v, a->q_codes, a->k_codes, a->v_codes, a->out, a->workspace};
    for (const void* p : al)
        if (!aligned16(p)) return HYQ_ERR_ALIGNMENT;
    return HYQ_OK;
}

static bool use_simt(const hyq_attn_args* a) { return a->impl == HYQ_IMPL_SIMT; }

// the tensor-core path of a planned call (arguments checked)
static int launch_planned(const hyq_attn_args& a, const TcPlan& plan, const TcSources* src, float alpha, cudaStream_t st) {
    if (!a.workspace || a.workspace_bytes < plan.w.total) return HYQ_ERR_WORKSPACE;
    return a.block_tokens == HYQ_BLOCK_TOKENS ? launch_attn_tc(a, plan, src, alpha, st) : tcbt::launch_attn_tc(a, plan, src, alpha, st);
}

int hyq_hybrid_attention_prefill_workspace(const hyq_attn_args* args, size_t* bytes) {
    if (!bytes) return HYQ_ERR_INVALID_ARG;
    const int rc = check_attn(args, false);
    if (rc != HYQ_OK) return rc;
    if (use_simt(args)) {
        *bytes = attn_simt_workspace_bytes(*args);
        return HYQ_OK;
    }
    TcPlan plan;
    if (!tc_plain_plan(*args, plan)) return HYQ_ERR_UNSUPPORTED;
    *bytes = tc_query_bytes(plan);
    return HYQ_OK;
}

int hyq_hybrid_attention_prefill(const hyq_attn_args* args, void* stream) {
    const int rc = check_attn(args, true);
    if (rc != HYQ_OK) return rc;
    const float alpha = args->softmax_scale != 0.0f ? args->softmax_scale : 1.0f / sqrtf((float)args->D);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (use_simt(args)) {
        const size_t need = attn_simt_workspace_bytes(*args);
        if (need > 0 && (!args->workspace || args->workspace_bytes < need)) return HYQ_ERR_WORKSPACE;
        return launch_attn_simt(*args, alpha, st);
    }
    TcPlan plan;
    if (!tc_plain_plan(*args, plan)) return HYQ_ERR_UNSUPPORTED;
    return launch_planned(*args, plan, nullptr, alpha, st);
}

// ---- ragged batches: the plain calls, sequence by sequence, on packed buffers ---------------------------------
static int check_cu(int n_seq, const int32_t* cu) {
    if (n_seq <= 0 || !cu || cu[0] != 0) return HYQ_ERR_INVALID_ARG;
    for (int s = 0; s < n_seq; ++s)
        if (cu[s + 1] <= cu[s]) return HYQ_ERR_INVALID_ARG;
    return HYQ_OK;
}

int hyq_select_vertical_varlen(const void* q_, const void* k_, int n_seq, const int32_t* cu, int Hq, int Hkv, int D,
                               int window, int n_tail, const int32_t* k_per_seq, int32_t* idx_out, void* workspace,
                               size_t workspace_bytes, void* stream) {
    int rc = check_cu(n_seq, cu);
    if (rc != HYQ_OK) return rc;
    if (!k_per_seq) return HYQ_ERR_INVALID_ARG;
    size_t need = 0;
    for (int s = 0; s < n_seq; ++s) {
        const int L = cu[s + 1] - cu[s];
        rc = check_select(q_, k_, 1, Hq, Hkv, L, L, D, window, n_tail, k_per_seq[s]);
        if (rc != HYQ_OK) return rc;
        const long P = L - window > 0 ? (long)L - window : 0;
        if (P > 0 && k_per_seq[s] > 0) need = need > select_workspace_bytes(1, Hq, L, window) ? need : select_workspace_bytes(1, Hq, L, window);
    }
    if (need == 0) return HYQ_OK;
    if (!q_ || !k_ || !idx_out || !workspace) return HYQ_ERR_INVALID_ARG;
    if (!aligned16(q_) || !aligned16(k_) || !aligned16(workspace) || (reinterpret_cast<uintptr_t>(idx_out) & 3u)) return HYQ_ERR_ALIGNMENT;
    if (workspace_bytes < need) return HYQ_ERR_WORKSPACE;
    // as many consecutive prompts per launch as the table and the workspace hold (each fits alone)
    size_t k_before = 0;
    for (int s = 0; s < n_seq && rc == HYQ_OK;) {
        SelTable tab;
        tab.early = 0;
        tab.n_seq = 0; tab.heads = Hq; tab.g = Hq / Hkv;
        for (; s < n_seq && tab.n_seq < SEL_MAX_SEQ; ++s) {
            const int L = cu[s + 1] - cu[s];
            SelSeq& q = tab.seq[tab.n_seq++] = SelSeq{};
            q.q = static_cast<const __nv_bfloat16*>(q_) + (size_t)Hq * D * cu[s];
            q.k = static_cast<const __nv_bfloat16*>(k_) + (size_t)Hkv * D * cu[s];
            q.Lq = q.Lk = L; q.t = n_tail ? n_tail : (window < L ? window : L);
            q.k_sel = L > window ? k_per_seq[s] : 0;
            q.P = q.k_sel > 0 ? L - window : 0;
            q.idx0 = (long)Hq * (long)k_before;
            if (tab.n_seq > 1 && select_scratch_bytes(tab) > workspace_bytes) { --tab.n_seq; break; }
            k_before += (size_t)k_per_seq[s];
        }
        rc = launch_select_table(tab, idx_out, workspace, static_cast<cudaStream_t>(stream));
    }
    return rc;
}

int hyq_quantize_blocks_varlen(const void* x, int n_seq, const int32_t* cu, int H, int D, int block_tokens, int format,
                               void* codes_out, float* scales_out, void* stream) {
    int rc = check_cu(n_seq, cu);
    if (rc != HYQ_OK) return rc;
    if (H <= 0 || !x || !codes_out || !scales_out) return HYQ_ERR_INVALID_ARG;
    if (D != HYQ_D || !block_tokens_ok(block_tokens)) return HYQ_ERR_UNSUPPORTED;
    if (format != HYQ_FMT_INT8 && format != HYQ_FMT_FP8_E4M3 && format != HYQ_FMT_INT4) return HYQ_ERR_UNSUPPORTED;
    if (!aligned16(x) || !aligned16(codes_out) || (reinterpret_cast<uintptr_t>(scales_out) & 3u)) return HYQ_ERR_ALIGNMENT;
    const size_t row_bytes = format == HYQ_FMT_INT4 ? D / 2 : D;
    size_t nb_before = 0;
    for (int s = 0; s < n_seq && rc == HYQ_OK;) {
        QuantJobs jobs;
        jobs.beside = 0;
        for (jobs.n = 0; s < n_seq && jobs.n < QUANT_MAX_JOBS; ++s) {
            const int L = cu[s + 1] - cu[s];
            QuantJob& j = jobs.job[jobs.n++] = QuantJob{};
            j.x = reinterpret_cast<const uint4*>(static_cast<const char*>(x) + (size_t)H * D * cu[s] * 2);
            j.codes = static_cast<uint8_t*>(codes_out) + (size_t)H * row_bytes * cu[s];
            j.scales = scales_out + (size_t)H * nb_before;
            j.L = L; j.heads = H; j.format = format;
            nb_before += (size_t)(L + block_tokens - 1) / block_tokens;
        }
        rc = launch_quantize_jobs(jobs, block_tokens, static_cast<cudaStream_t>(stream));
    }
    return rc;
}

// Plan of the consecutive sequences [s0, s0 + n) of a ragged call as one launch; their packed buffers' first bytes in `a`.
// False when one launch cannot hold them.
static bool plan_group(const hyq_attn_args& args, int s0, int n, const int32_t* cu, const int32_t* k_per_seq, TcPlan& plan) {
    if (n > TC_MAX_SEQ) return false;
    TcSeq seq[TC_MAX_SEQ];
    size_t k_before = 0, nb_before = 0;
    for (int i = 0; i < n; ++i) {
        const int L = cu[s0 + i + 1] - cu[s0 + i];
        seq[i] = tc_ragged_seq(args, L, k_per_seq[s0 + i], (size_t)(cu[s0 + i] - cu[s0]), k_before, nb_before);
        k_before += (size_t)k_per_seq[s0 + i];
        nb_before += (size_t)((L + args.block_tokens - 1) / args.block_tokens);
    }
    return tc_make_plan(args, seq, n, args.Hq, args.Hq / args.Hkv, plan);
}
// the largest group of sequences from s0 on that one launch within `bytes` of workspace can hold (halved until it fits)
static int next_group(const hyq_attn_args& args, int s0, int n_seq, const int32_t* cu, const int32_t* k_per_seq, size_t bytes, TcPlan& plan) {
    int n = n_seq - s0 < TC_MAX_SEQ ? n_seq - s0 : TC_MAX_SEQ;
    while (!(plan_group(args, s0, n, cu, k_per_seq, plan) && plan.w.total <= bytes)) {
        if (n == 1) return 0;
        n = (n + 1) / 2;
    }
    return n;
}

// the arguments of the sequences from s on: packed pointers advanced to sequence s
static hyq_attn_args at_sequence(const hyq_attn_args& args, int L, int k, size_t t0, size_t k_before, size_t nb_before) {
    const size_t q_row = args.q_format == HYQ_FMT_INT4 ? HYQ_D / 2 : HYQ_D, k_row = args.k_format == HYQ_FMT_INT4 ? HYQ_D / 2 : HYQ_D;
    const size_t v_row = args.v_format == HYQ_FMT_INT4 ? HYQ_D / 2 : HYQ_D;
    hyq_attn_args a = args;
    a.B = 1; a.L = L; a.Lq = 0; a.k = k;
    auto at = [](const void* base, size_t bytes) -> const void* { return base ? static_cast<const char*>(base) + bytes : nullptr; };
    a.q = at(args.q, (size_t)args.Hq * HYQ_D * t0 * 2);
    a.k_ = at(args.k_, (size_t)args.Hkv * HYQ_D * t0 * 2);
    a.v = at(args.v, (size_t)args.Hkv * HYQ_D * t0 * 2);
    a.q_codes = at(args.q_codes, (size_t)args.Hq * q_row * t0);
    a.k_codes = at(args.k_codes, (size_t)args.Hkv * k_row * t0);
    a.v_codes = at(args.v_codes, (size_t)args.Hkv * v_row * t0);
    a.q_scales = args.q_scales ? args.q_scales + (size_t)args.Hq * nb_before : nullptr;
    a.k_scales = args.k_scales ? args.k_scales + (size_t)args.Hkv * nb_before : nullptr;
    a.v_scales = args.v_scales ? args.v_scales + (size_t)args.Hkv * nb_before : nullptr;
    a.vl_idx = args.vl_idx ? args.vl_idx + (size_t)args.Hq * k_before : nullptr;
    a.out = const_cast<void*>(at(args.out, (size_t)args.Hq * HYQ_D * t0 * (args.out_dtype == 1 ? 4 : 2)));
    a.lse = args.lse ? args.lse + (size_t)args.Hq * t0 : nullptr;
    return a;
}

int hyq_hybrid_attention_prefill_varlen_workspace(const hyq_attn_args* args, int n_seq, const int32_t* cu, const int32_t* k_per_seq,
                                                  size_t* bytes) {
    int rc = check_cu(n_seq, cu);
    if (rc != HYQ_OK) return rc;
    if (!bytes || !k_per_seq || !args || args->struct_size != sizeof(hyq_attn_args)) return HYQ_ERR_INVALID_ARG;
    size_t most = 0;
    TcPlan plan;
    for (int s = 0; s < n_seq && rc == HYQ_OK; ++s) {
        const int L = cu[s + 1] - cu[s];
        hyq_attn_args a = at_sequence(*args, L, k_per_seq[s], 0, 0, 0);
        if (a.k < 0 || a.k > (L - a.window > 0 ? L - a.window : 0)) return HYQ_ERR_INVALID_ARG;
        rc = check_attn(&a, false);
        if (rc == HYQ_OK && use_simt(&a) && attn_simt_workspace_bytes(a) > most) most = attn_simt_workspace_bytes(a);
    }
    if (rc != HYQ_OK || use_simt(args)) { *bytes = most; return rc; }
    for (int s = 0, n; s < n_seq; s += n) {
        n = next_group(*args, s, n_seq, cu, k_per_seq, (size_t)-1, plan);
        if (n == 0) return HYQ_ERR_UNSUPPORTED;
        if (plan.w.total > most) most = plan.w.total;
    }
    *bytes = most;
    return HYQ_OK;
}

int hyq_hybrid_attention_prefill_varlen(const hyq_attn_args* args, int n_seq, const int32_t* cu, const int32_t* k_per_seq,
                                        void* stream) {
    int rc = check_cu(n_seq, cu);
    if (rc != HYQ_OK) return rc;
    if (!args || args->struct_size != sizeof(hyq_attn_args) || !k_per_seq) return HYQ_ERR_INVALID_ARG;
    const int bt = args->block_tokens;
    if (!block_tokens_ok(bt)) return HYQ_ERR_UNSUPPORTED;
    // every sequence is checked, alone, before the first launch: any of them fits the workspace by itself
    TcPlan plan;
    size_t nb_before = 0, k_before = 0;
    for (int s = 0; s < n_seq && rc == HYQ_OK; ++s) {
        const int L = cu[s + 1] - cu[s];
        const hyq_attn_args a = at_sequence(*args, L, k_per_seq[s], (size_t)cu[s], k_before, nb_before);
        if (a.k < 0 || a.k > (L - a.window > 0 ? L - a.window : 0)) rc = HYQ_ERR_INVALID_ARG;
        if (rc == HYQ_OK) rc = check_attn(&a, true);
        if (rc == HYQ_OK) {
            if (!use_simt(&a) && !plan_group(*args, s, 1, cu, k_per_seq, plan)) rc = HYQ_ERR_UNSUPPORTED;
            const size_t need = use_simt(&a) ? attn_simt_workspace_bytes(a) : plan.w.total;
            if (rc == HYQ_OK && need > 0 && (!a.workspace || a.workspace_bytes < need)) rc = HYQ_ERR_WORKSPACE;
        }
        nb_before += (size_t)(L + bt - 1) / bt;
        k_before += (size_t)k_per_seq[s];
    }
    const float alpha = args->softmax_scale != 0.0f ? args->softmax_scale : 1.0f / sqrtf((float)args->D);
    nb_before = k_before = 0;
    for (int s = 0, n; s < n_seq && rc == HYQ_OK; s += n) {
        const hyq_attn_args a = at_sequence(*args, cu[s + 1] - cu[s], k_per_seq[s], (size_t)cu[s], k_before, nb_before);
        if (use_simt(&a)) {
            n = 1;
            rc = launch_attn_simt(a, alpha, static_cast<cudaStream_t>(stream));
        } else {
            n = next_group(*args, s, n_seq, cu, k_per_seq, args->workspace_bytes, plan);
            rc = n > 0 ? launch_planned(a, plan, nullptr, alpha, static_cast<cudaStream_t>(stream)) : HYQ_ERR_WORKSPACE;
        }
        for (int i = s; i < s + n; ++i) {
            nb_before += (size_t)(cu[i + 1] - cu[i] + bt - 1) / bt;
            k_before += (size_t)k_per_seq[i];
        }
    }
    return rc;
}

// ---- the whole path in one call ---------------------------------------------------------------------------------
// the attention arguments of the sequences from s on (offsets in tokens / indices / blocks of the packed results)
static hyq_attn_args attn_args_of(const hyq_prefill_args& a, int s, size_t t0, size_t k_before, size_t nb_before) {
    hyq_attn_args x{};
    x.struct_size = sizeof(x);
    x.B = a.B; x.Hq = a.Hq; x.Hkv = a.Hkv; x.L = a.lengths[s]; x.D = a.D;
    x.window = a.window; x.k = a.k_per_seq[s]; x.block_tokens = a.block_tokens;
    x.q_format = a.q_format; x.k_format = a.k_format; x.v_format = a.v_format;
    x.out_dtype = a.out_dtype; x.softmax_scale = a.softmax_scale;
    x.q = a.q ? a.q[s] : nullptr; x.k_ = a.k_ ? a.k_[s] : nullptr; x.v = a.v ? a.v[s] : nullptr;
    auto row = [](int fmt) -> size_t { return fmt == HYQ_FMT_INT4 ? HYQ_D / 2 : HYQ_D; };
    auto at = [](const void* base, size_t bytes) -> const void* { return base ? static_cast<const char*>(base) + bytes : nullptr; };
    x.q_codes = at(a.q_codes, a.Hq * row(a.q_format) * t0);
    x.k_codes = at(a.k_codes, a.Hkv * row(a.k_format) * t0);
    x.v_codes = at(a.v_codes, a.Hkv * row(a.v_format) * t0);
    x.q_scales = a.q_scales ? a.q_scales + a.Hq * nb_before : nullptr;
    x.k_scales = a.k_scales ? a.k_scales + a.Hkv * nb_before : nullptr;
    x.v_scales = a.v_scales ? a.v_scales + a.Hkv * nb_before : nullptr;
    x.vl_idx = a.idx ? a.idx + a.Hq * k_before : nullptr;
    x.out = const_cast<void*>(at(a.out, (size_t)a.Hq * HYQ_D * t0 * (a.out_dtype == 1 ? 4 : 2)));
    x.lse = a.lse ? a.lse + a.Hq * t0 : nullptr;
    x.status_word = a.status_word;
    x.workspace = a.workspace; x.workspace_bytes = a.workspace_bytes;
    return x;
}

static int check_prefill(const hyq_prefill_args* a, bool need_pointers) {
    if (!a || a->struct_size != sizeof(hyq_prefill_args) || a->n_seq <= 0 || !a->lengths || !a->k_per_seq) return HYQ_ERR_INVALID_ARG;
    if (a->B <= 0 || (a->B > 1 && a->n_seq > 1)) return HYQ_ERR_INVALID_ARG;
    if (need_pointers && (!a->q || !a->k_ || !a->v)) return HYQ_ERR_INVALID_ARG;
    if (!block_tokens_ok(a->block_tokens)) return HYQ_ERR_UNSUPPORTED;
    if (need_pointers && ((reinterpret_cast<uintptr_t>(a->idx) | reinterpret_cast<uintptr_t>(a->q_scales) |
                           reinterpret_cast<uintptr_t>(a->k_scales) | reinterpret_cast<uintptr_t>(a->v_scales)) & 3u))
        return HYQ_ERR_ALIGNMENT;
    size_t t0 = 0, k0 = 0, nb0 = 0;
    for (int s = 0; s < a->n_seq; ++s) {
        const int L = a->lengths[s];
        int rc = check_select(nullptr, nullptr, a->B, a->Hq, a->Hkv, L, L, a->D, a->window, a->n_tail, a->k_per_seq[s]);
        if (rc != HYQ_OK) return rc;
        if (a->k_per_seq[s] > (L - a->window > 0 ? L - a->window : 0)) return HYQ_ERR_INVALID_ARG;
        const hyq_attn_args x = attn_args_of(*a, s, t0, k0, nb0);
        rc = check_attn(&x, need_pointers);
        if (rc != HYQ_OK) return rc;
        t0 += (size_t)L; k0 += (size_t)a->k_per_seq[s]; nb0 += (size_t)((L + a->block_tokens - 1) / a->block_tokens);
    }
    return HYQ_OK;
}

// what one round of launches needs: sequences [s, s + n) of a call
struct PrefillGroup {
    TcPlan plan;
    SelTable sel;
    size_t sel_at, total;
};
static bool plan_prefill(const hyq_prefill_args& a, int s, int n, PrefillGroup& g) {
    const hyq_attn_args x = attn_args_of(a, s, 0, 0, 0);
    TcSeq seq[TC_MAX_SEQ];
    size_t t0 = 0, k0 = 0, nb0 = 0;
    g.sel.n_seq = n; g.sel.heads = a.B * a.Hq; g.sel.g = a.Hq / a.Hkv;
    for (int i = 0; i < n; ++i) {
        const int L = a.lengths[s + i], k = a.k_per_seq[s + i];
        seq[i] = tc_ragged_seq(x, L, k, t0, k0, nb0);
        SelSeq& q = g.sel.seq[i] = SelSeq{};
        q.q = a.q ? static_cast<const __nv_bfloat16*>(a.q[s + i]) : nullptr;
        q.k = a.k_ ? static_cast<const __nv_bfloat16*>(a.k_[s + i]) : nullptr;
        q.Lq = q.Lk = L; q.t = a.n_tail ? a.n_tail : (a.window < L ? a.window : L);
        q.P = k > 0 && L > a.window ? L - a.window : 0;
        q.k_sel = k; q.idx0 = (long)a.Hq * (long)k0;
        t0 += (size_t)L; k0 += (size_t)k; nb0 += (size_t)((L + a.block_tokens - 1) / a.block_tokens);
    }
    if (!tc_make_plan(x, seq, n, a.B * a.Hq, a.Hq / a.Hkv, g.plan)) return false;
    g.sel_at = align_up(g.plan.w.total, 256);
    g.total = g.sel_at + select_scratch_bytes(g.sel);
    return true;
}
// as many sequences from s on as one round of launches within `bytes` of workspace can hold (halved until it fits; 0: not one)
static int next_prefill_group(const hyq_prefill_args& a, int s, size_t bytes, PrefillGroup& g) {
    int n = a.n_seq - s < TC_MAX_SEQ ? a.n_seq - s : TC_MAX_SEQ;
    while (!(plan_prefill(a, s, n, g) && g.total <= bytes)) {
        if (n == 1) return 0;
        n = (n + 1) / 2;
    }
    return n;
}

int hyq_hybrid_prefill_workspace(const hyq_prefill_args* args, size_t* bytes) {
    if (!bytes) return HYQ_ERR_INVALID_ARG;
    const int rc = check_prefill(args, false);
    if (rc != HYQ_OK) return rc;
    size_t most = 0;
    PrefillGroup g;
    for (int s = 0, n; s < args->n_seq; s += n) {
        n = next_prefill_group(*args, s, (size_t)-1, g);
        if (n == 0) return HYQ_ERR_UNSUPPORTED;
        most = g.total > most ? g.total : most;
    }
    *bytes = most;
    return HYQ_OK;
}

constexpr size_t BESIDE_BYTES = (size_t)256 << 20;
int hyq_hybrid_prefill(const hyq_prefill_args* args, void* stream) {
    int rc = check_prefill(args, true);
    if (rc != HYQ_OK) return rc;
    const hyq_prefill_args& a = *args;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PrefillGroup g;
    if (!a.workspace) return HYQ_ERR_INVALID_ARG;
    if (a.n_seq > 1)                                            // (one sequence: its only group below says so)
        for (int s = 0; s < a.n_seq; ++s)
            if (!plan_prefill(a, s, 1, g) || g.total > a.workspace_bytes) return HYQ_ERR_WORKSPACE;
    const float alpha = a.softmax_scale != 0.0f ? a.softmax_scale : 1.0f / sqrtf((float)a.D);
    size_t t0 = 0, k0 = 0, nb0 = 0;
    for (int s = 0, n; s < a.n_seq; s += n) {
        n = next_prefill_group(a, s, a.workspace_bytes, g);
        if (n == 0) return HYQ_ERR_WORKSPACE;
        const hyq_attn_args x = attn_args_of(a, s, t0, k0, nb0);
        char* base = static_cast<char*>(a.workspace);
        QuantJobs jobs;
        TcSources src;
        jobs.n = 3 * n;
        bool selects = false;
        size_t tt = 0, nb = 0;
        for (int i = 0; i < n; ++i) {
            const int L = a.lengths[s + i];
            src.q[i] = a.q[s + i]; src.k[i] = a.k_[s + i]; src.v[i] = a.v[s + i];
            auto job = [&](int which, const void* data, int H, int format, const void* codes, const float* scales) -> QuantJob& {
                QuantJob& j = jobs.job[3 * i + which] = QuantJob{};
                const size_t row = format == HYQ_FMT_INT4 ? HYQ_D / 2 : HYQ_D;
                j.x = static_cast<const uint4*>(data); j.L = L; j.heads = a.B * H; j.format = format;
                j.codes = static_cast<uint8_t*>(const_cast<void*>(codes)) + H * row * tt;
                j.scales = const_cast<float*>(scales) + H * nb;
                return j;
            };
            QuantJob& jq = job(0, a.q[s + i], a.Hq, a.q_format, x.q_codes, x.q_scales);
            QuantJob& jk = job(1, a.k_[s + i], a.Hkv, a.k_format, x.k_codes, x.k_scales);
            QuantJob& jv = job(2, a.v[s + i], a.Hkv, a.v_format, x.v_codes, x.v_scales);
            if (a.q_format == HYQ_FMT_INT4) {
                jq.wide = reinterpret_cast<uint8_t*>(base + g.plan.w.q8) + a.Hq * tt * HYQ_D;
                jk.wide = reinterpret_cast<uint8_t*>(base + g.plan.w.k8) + a.Hkv * tt * HYQ_D;
            }
            jv.v16 = reinterpret_cast<uint4*>(base + g.plan.w.v16) + a.Hkv * tt * (HYQ_D / 8);
            jv.vh16 = reinterpret_cast<uint4*>(base + g.plan.w.vh16) + a.Hkv * tt * (HYQ_D / 8);
            jk.kv_fac = jv.kv_fac = reinterpret_cast<float4*>(base + g.plan.w.kv_fac) + a.Hkv * nb;
            tt += (size_t)L; nb += (size_t)((L + a.block_tokens - 1) / a.block_tokens);
            k0 += (size_t)a.k_per_seq[s + i];
            selects |= g.sel.seq[i].P > 0 && g.sel.seq[i].k_sel > 0;          // (the selection launches something)
        }
        // Neither needs the other: the quantizer, which moves memory, runs beside the selection's three kernels, which wait for
        // latencies and the fp64 pipe (2 heads x 2048 tokens 45.5 -> 42.8 us a call, eight prompts with 0.2 GB of Q, K and V 624 -> 616).
        // Where both fill the GPU for long they only get in each other's way: 0.4 GB 6861 -> 6863 us, 0.9 GB 9924 -> 9977.
        const bool beside = selects && 2 * (size_t)a.B * (a.Hq + 2 * a.Hkv) * tt * HYQ_D <= BESIDE_BYTES;
        jobs.beside = g.sel.early = beside;
        if (!beside) rc = launch_quantize_jobs(jobs, a.block_tokens, st);
        if (rc == HYQ_OK) rc = launch_select_table(g.sel, const_cast<int32_t*>(x.vl_idx), base + g.sel_at, st);
        if (rc == HYQ_OK && beside) rc = launch_quantize_jobs(jobs, a.block_tokens, st);
        if (rc == HYQ_OK) rc = launch_planned(x, g.plan, &src, alpha, st);
        if (rc != HYQ_OK) return rc;
        t0 += tt; nb0 += nb;
    }
    return HYQ_OK;
}

}  // extern "C"

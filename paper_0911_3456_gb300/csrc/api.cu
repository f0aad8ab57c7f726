// api.cu -- the C ABI of libfbcorr: plan creation, variant selection,
// forward / backward dispatch and the auto-tuner.
//
// Control flow mirrors the paper's RTCG loop (Fig. 1, Sec. 6.2): a plan
// fixes the problem shape, code is generated and compiled for exactly that
// shape (NVRTC, cached), candidates are timed when tuning is requested and the
// winner is remembered per GPU and shape; the per-call path is then a single
// prepared launch.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <sstream>

#include "internal.h"

namespace fbc {
const char* last_error_message();
}

using namespace fbc;

namespace {

// Host mirror of the NVRTC dL/dw kernel's by-value argument struct (rtcg_direct.cuh).
struct DwArgsK {
    const float* x;
    const float* g;
    const float* m;
    float* part;
    int H, W, Ho, Wo, N;
    int rows_per_chunk;
    float lo, hi;
    const int* flags;
    int nflags;
};

const int64_t kMaxElems = (int64_t)1 << 31;

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

DirectProblem fwd_problem(const fbcorr_plan* p) {
    DirectProblem pr;
    pr.in_h = (int)p->H;
    pr.in_w = (int)p->W;
    pr.c = (int)p->D;
    pr.out_h = (int)p->Ho;
    pr.out_w = (int)p->Wo;
    pr.nf = (int)p->N;
    pr.fh = (int)p->fh;
    pr.fw = (int)p->fw;
    pr.pad_y = 0;
    pr.pad_x = 0;
    pr.flip = 0;
    pr.epi = p->epi.kind == FBCORR_EPI_CLAMP ? 1 : (p->epi.kind == FBCORR_EPI_SNIPPET ? 2 : 0);
    pr.mask = 0;
    pr.snippet = p->snippet;
    return pr;
}

DirectProblem dx_problem(const fbcorr_plan* p) {
    DirectProblem pr;
    pr.in_h = (int)p->Ho;
    pr.in_w = (int)p->Wo;
    pr.c = (int)p->N;
    pr.out_h = (int)p->H;
    pr.out_w = (int)p->W;
    pr.nf = (int)p->D;
    pr.fh = (int)p->fh;
    pr.fw = (int)p->fw;
    pr.pad_y = (int)p->fh - 1;
    pr.pad_x = (int)p->fw - 1;
    pr.flip = 1;
    pr.epi = 0;
    pr.mask = p->epi.kind == FBCORR_EPI_CLAMP ? 1 : 0;
    return pr;
}

const char* kind_name(VarKind k) {
    switch (k) {
        case VarKind::Default: return "default";
        case VarKind::Direct: return "direct";
        case VarKind::Tensor: return "tcgen05";
        case VarKind::F32tc: return "f32tc";
    }
    return "?";
}

std::string shape_key(const fbcorr_plan* p, const char* what) {
    std::ostringstream o;
    o << what << "|x" << p->H << "x" << p->W << "x" << p->D << "|w" << p->N << "x" << p->fh << "x"
      << p->fw << "|dt" << (int)p->dtype << "|epi" << p->epi.kind;
    return o.str();
}

// The spec of the variant an untuned FP32 problem takes: the tensor-core kernel
// where the model expects it to win over the FMA kernels.
std::string heuristic_spec(const DirectProblem& pr, const DeviceInfo& dev) {
    F3Tile f3;
    if (f3_wins(pr, dev.sm_count, &f3)) return f3_spec(f3);
    return direct_tile_spec(direct_heuristic(pr, smem_limit(dev), dev.sm_count));
}

// BF16 modes: the packed kernel with tile t instead of the plan's own tensor-core kernel.
int plan_orders(const fbcorr_plan* p) { return p->dtype == FBCORR_F32 ? 3 : p->dtype == FBCORR_BF16X3 ? 2 : 1; }

fbcorr_status_t set_packed(fbcorr_plan* p, const F3Tile& t, const char* source) {
    const DirectProblem pr = fwd_problem(p);
    if (f3_ws_bytes(pr, t) > p->ws_fwd)
        return set_error(FBCORR_ERR_UNSUPPORTED, "variant %s needs more workspace than the plan's", f3_spec(t).c_str());
    F3Launch l;
    FBC_TRY(f3_build(pr, t, p->dev.sm_count, &l));
    p->fwd_f3 = l;
    p->tc_packed = true;
    p->fwd_source = source;
    return FBCORR_OK;
}

// Select the forward variant of a BF16 or split-BF16 plan from a spec string.
fbcorr_status_t set_tc_spec(fbcorr_plan* p, const std::string& spec, const char* source) {
    F3Tile t;
    if (f3_parse_spec(spec, &t, plan_orders(p))) return set_packed(p, t, source);
    FBC_TRY(tc_set_spec(p->tc, spec));
    p->tc_packed = false;
    p->fwd_source = source;
    return FBCORR_OK;
}

// The variant of an untuned BF16 or split-BF16 plan, whose tc is at its default.
fbcorr_status_t set_tc_heuristic(fbcorr_plan* p) {
    p->tc_packed = false;
    p->fwd_source = "heuristic";
    F3Tile t;
    if (f3_wins_bf16(fwd_problem(p), p->dev.sm_count, plan_orders(p), p->ws_fwd, &t) &&
        set_packed(p, t, "heuristic") != FBCORR_OK)
        logf("packed tensor-core kernel not usable (%s)", last_error_message());
    return FBCORR_OK;
}

// The FMA kernel that calls without scratch run beside a tensor-core one (what: "fwd"
// or "dx"): the spec `fma`, the tuning cache's, or the heuristic's, whichever is the
// first to fit.  The prebuilt kernel ("default") is an empty *k.
fbcorr_status_t build_fma(const fbcorr_plan* p, const char* what, const DirectProblem& pr, std::string fma, DirectTile* t,
                          Kernel* k) {
    *k = Kernel{};
    if (!fma.empty() || tune_lookup(tune_key(p->dev, shape_key(p, what) + "|fma"), &fma)) {
        if (fma == "default" && p->snippet.empty()) return FBCORR_OK;
        if (parse_direct_spec(fma, t) && direct_smem_bytes(*t, pr.fh, pr.fw, pr.c) <= smem_limit(p->dev) &&
            build_direct(pr, *t, k) == FBCORR_OK)
            return FBCORR_OK;
        logf("FMA variant '%s' not usable; ignoring it", fma.c_str());
    }
    *t = direct_heuristic(pr, smem_limit(p->dev), p->dev.sm_count);
    return build_direct(pr, *t, k);
}

fbcorr_status_t run_fma(const Kernel& k, const DirectTile& t, const DirectProblem& pr, const float* x, const float* m,
                        const float* w, float* y, float lo, float hi, cudaStream_t s) {
    return k.fn ? run_direct(k, pr, t, x, m, w, y, lo, hi, s) : run_default(pr, x, m, w, y, lo, hi, s);
}

// Select the forward variant of an F32 plan from a spec string (fma: see build_fma).
fbcorr_status_t set_fwd_spec(fbcorr_plan* p, const std::string& spec, const char* source, const std::string& fma = "") {
    if (spec == "default" && !p->snippet.empty())
        return set_error(FBCORR_ERR_UNSUPPORTED, "the prebuilt default kernel has no snippet epilogue");
    if (spec == "default") {
        p->fwd_kind = VarKind::Default;
        p->fwd_kernel = Kernel{};
        p->fwd_source = source;
        return FBCORR_OK;
    }
    const DirectProblem pr = fwd_problem(p);
    F3Tile f3;
    if (f3_parse_spec(spec, &f3)) {
        F3Launch l;
        FBC_TRY(f3_build(pr, f3, p->dev.sm_count, &l));
        DirectTile dt;
        Kernel k;
        FBC_TRY(build_fma(p, "fwd", pr, fma, &dt, &k));
        p->fwd_kind = VarKind::F32tc;
        p->fwd_f3 = l;
        p->fwd_tile = dt;
        p->fwd_kernel = k;
        p->fwd_source = source;
        return FBCORR_OK;
    }
    DirectTile t;
    if (!parse_direct_spec(spec, &t))
        return set_error(FBCORR_ERR_INVALID_ARG, "unknown variant spec '%s'", spec.c_str());
    if (direct_smem_bytes(t, pr.fh, pr.fw, pr.c) > smem_limit(p->dev))
        return set_error(FBCORR_ERR_UNSUPPORTED, "variant %s needs too much shared memory",
                         spec.c_str());
    Kernel k;
    FBC_TRY(build_direct(pr, t, &k));
    p->fwd_kind = VarKind::Direct;
    p->fwd_tile = t;
    p->fwd_kernel = k;
    p->fwd_source = source;
    return FBCORR_OK;
}

fbcorr_status_t choose_fwd_f32(fbcorr_plan* p) {
    const std::string env = env_str("FBCORR_VARIANT", "");
    if (!env.empty()) {
        fbcorr_status_t s = set_fwd_spec(p, env, "env");
        if (s == FBCORR_OK) return s;
        logf("FBCORR_VARIANT=%s not usable (%s); continuing", env.c_str(), last_error_message());
    }
    std::string cached;
    if (tune_lookup(tune_key(p->dev, shape_key(p, "fwd")), &cached)) {
        if (set_fwd_spec(p, cached, "cache") == FBCORR_OK) return FBCORR_OK;
        logf("tune-cache entry '%s' not usable; ignoring it", cached.c_str());
    }
    fbcorr_status_t s = set_fwd_spec(p, heuristic_spec(fwd_problem(p), p->dev), "heuristic");
    if (s == FBCORR_ERR_NVRTC && p->snippet.empty()) {
        logf("code generation failed, falling back to the prebuilt default kernel: %s",
             last_error_message());
        return set_fwd_spec(p, "default", "fallback");
    }
    return s;
}

// Row chunks of the generated dL/dw kernel once its residency is known: the
// launch runs fh x filter-block x chunk CTAs, `resident` per SM at a time, each
// over rows_per_chunk output rows, so its length goes as (rounds of resident
// CTAs) x rows_per_chunk.  Take the fewest rows per chunk that minimise that
// product, never more chunks than the workspace planned at creation holds
// (e.g. 250 rows, 7 filter rows, 3 CTAs per SM on 152 SMs: 63 chunks of 4 rows
// in one round instead of 84 chunks of 3 rows in two).
void replan_dw_chunks(fbcorr_plan* p, int resident) {
    const long slots = (long)std::max(1, p->dev.sm_count) * resident;
    const long per_chunk = (long)p->fh * p->dw_nblocks;
    int best_rows = p->dw_rows_per_chunk;
    long best = -1;
    for (int rows = p->dw_rows_per_chunk; rows <= p->Ho; ++rows) {
        const long chunks = (p->Ho + rows - 1) / rows;
        const long rounds = (chunks * per_chunk + slots - 1) / slots;
        const long cost = rounds * rows;
        if (best < 0 || cost < best) {
            best = cost;
            best_rows = rows;
        }
    }
    p->dw_rows_per_chunk = best_rows;
    p->dw_chunks = (int)((p->Ho + best_rows - 1) / best_rows);
}

// The dL/dx variant: forced (tests, profiling), tuned, or the model's.
std::string dx_spec(const fbcorr_plan* p) {
    std::string spec = env_str("FBCORR_DX_VARIANT", "");
    if (!spec.empty() || tune_lookup(tune_key(p->dev, shape_key(p, "dx")), &spec)) return spec;
    return heuristic_spec(dx_problem(p), p->dev);
}

// The forward problem with the mask of dL/dw.
DirectProblem dw_problem(const fbcorr_plan* p) {
    DirectProblem pr = fwd_problem(p);
    pr.epi = 0;
    pr.mask = p->epi.kind == FBCORR_EPI_CLAMP ? 1 : 0;
    return pr;
}

// A backward workspace with scratch: the FMA kernel's dL/dw partial sums, the dL/dx
// scratch, the tensor-core kernel's dL/dw partial sums.
size_t dx_scratch_offset(const fbcorr_plan* p) { return (p->ws_bwd + 255) / 256 * 256; }
size_t dw_scratch_offset(const fbcorr_plan* p) {
    return (dx_scratch_offset(p) + (p->dx_kind == VarKind::F32tc ? p->dx_f3.ws_bytes : 0) + 255) / 256 * 256;
}

fbcorr_status_t prepare_backward(fbcorr_plan* p) {
    if (p->bwd_ready) return FBCORR_OK;
    const DirectProblem pr = dx_problem(p);
    DirectTile t = direct_heuristic(pr, smem_limit(p->dev), p->dev.sm_count);
    const std::string spec = dx_spec(p);
    const bool use_default = spec == "default";
    DirectTile ct;
    if (parse_direct_spec(spec, &ct) && direct_smem_bytes(ct, pr.fh, pr.fw, pr.c) <= smem_limit(p->dev)) t = ct;
    Kernel k;
    F3Tile f3;
    F3Launch l;
    // with scratch the tensor-core kernel runs, without it the FMA kernel
    const bool tensor = f3_parse_spec(spec, &f3) && f3_build(pr, f3, p->dev.sm_count, &l) == FBCORR_OK;
    fbcorr_status_t s = use_default ? FBCORR_ERR_NVRTC : tensor ? build_fma(p, "dx", pr, "", &t, &k) : build_direct(pr, t, &k);
    if (s == FBCORR_OK) {
        p->dx_kind = tensor ? VarKind::F32tc : VarKind::Direct;
        p->dx_tile = t;
        p->dx_kernel = k;
        p->dx_f3 = l;
    } else if (s == FBCORR_ERR_NVRTC) {
        p->dx_kind = VarKind::Default;
    } else {
        return s;
    }
    const int mask = p->epi.kind == FBCORR_EPI_CLAMP ? 1 : 0;
    if (p->D > 256) {
        p->dw_kind = VarKind::Default;   // one thread per channel does not fit a CTA
    } else {
        char name[160];
        // FMA form, chosen with the tile at plan creation (FBCORR_DW_PK): 0 scalar;
        // 1 packed pairs with register totals (about 120 registers); 2 (default)
        // packed pairs with the chunk totals in shared memory
        if (p->dw_pk == 2 &&
            dw_smem_bytes((int)p->fw, (int)p->D, p->dw_tn, p->dw_ng, p->dw_qb, 2) > smem_limit(p->dev))
            p->dw_pk = 0;   // the totals do not fit beside the buffers
        // launch bounds: as many CTAs per SM (at most 3) as the shared memory
        // holds, so that the register allocator keeps that residency
        const size_t need = dw_smem_bytes((int)p->fw, (int)p->D, p->dw_tn, p->dw_ng, p->dw_qb, p->dw_pk);
        const size_t per_sm = 228 * 1024;   // shared memory per SM (sm_100 family)
        p->dw_mb = std::max(1, std::min(3, (int)(per_sm / (need + 1024))));
        const int mb_env = atoi(env_str("FBCORR_DW_MB", "-1").c_str());
        if (mb_env >= 0 && mb_env <= 4) p->dw_mb = mb_env;   // 0: no launch bound
        auto build_dw = [&]() {
            snprintf(name, sizeof name, "fbc_dw_f%dx%d_c%d_n%d_g%d_q%d_m%d%s_b%d", (int)p->fh, (int)p->fw,
                     (int)p->D, p->dw_tn, p->dw_ng, p->dw_qb, mask,
                     p->dw_pk == 1 ? "_pk1" : p->dw_pk == 2 ? "_pk2" : "", p->dw_mb);
            return rtcg_kernel(dw_kernel_source((int)p->fh, (int)p->fw, (int)p->D, p->dw_tn, p->dw_ng,
                                                p->dw_qb, mask, p->dw_pk, name, p->dw_mb),
                               name, need, (int)p->D * p->dw_ng, &p->dw_kernel);
        };
        s = build_dw();
        int regs = 0, local = 0;
        if (s == FBCORR_OK && p->dw_mb > 0 && mb_env < 0 &&
            kernel_resources(p->dw_kernel, &regs, &local) == FBCORR_OK && local > 0) {
            p->dw_mb = 0;   // the bound made the allocator spill (wide filters): drop it
            s = build_dw();
        }
        if (s == FBCORR_OK) {
            p->dw_kind = VarKind::Direct;
            F3DwTile dt;
            F3DwLaunch dl;
            p->dw_f3 = F3DwLaunch{};
            if (f3dw_wins(dw_problem(p), p->dev.sm_count, &dt) && f3dw_build(dw_problem(p), dt, &dl) == FBCORR_OK)
                p->dw_f3 = dl;
            if (kernel_resources(p->dw_kernel, &regs, &local) == FBCORR_OK) p->dw_regs = regs;
            int resident = 0;
            if (kernel_occupancy(p->dw_kernel, &resident) == FBCORR_OK && resident > 0)
                replan_dw_chunks(p, resident);
        } else if (s == FBCORR_ERR_NVRTC) {
            p->dw_kind = VarKind::Default;
        } else {
            return s;
        }
    }
    if (!p->bwd_side) {
        // side stream for dL/dw when both gradients are wanted; without it the two
        // run one after the other on the caller's stream
        if (cudaStreamCreateWithFlags(&p->bwd_side, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&p->bwd_fork, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&p->bwd_join, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            if (p->bwd_side) cudaStreamDestroy(p->bwd_side);
            if (p->bwd_fork) cudaEventDestroy(p->bwd_fork);
            if (p->bwd_join) cudaEventDestroy(p->bwd_join);
            p->bwd_side = nullptr;
            p->bwd_fork = p->bwd_join = nullptr;
        }
    }
    p->bwd_ready = true;
    return FBCORR_OK;
}

void plan_dw_chunks(fbcorr_plan* p) {
    // CTA = NG filter groups x D channels (about 256 threads with 4 filters per
    // thread, 128 with 8); enough row chunks for about 4 resident CTAs per SM
    // over two waves (re-planned from the built kernel's residency); deterministic
    // in the shape
    // FMA form (FBCORR_DW_PK, default 2): packed pairs with the chunk totals in
    // shared memory.  Measured on the differentiation workload (256x256x16 input,
    // 64 filters 7x7x16): scalar 0.149 ms, packed pairs with register totals (2
    // CTAs per SM) 0.143, with shared totals 0.132 (4 filters per thread) and
    // 0.130 (8 filters per thread, 128-thread CTAs, 3 per SM).
    const std::string pk_env = env_str("FBCORR_DW_PK", "2");
    p->dw_pk = pk_env == "1" ? 1 : pk_env == "0" ? 0 : 2;
    // 8 filters per thread where the packed double-buffered path runs (16-byte
    // rows of g and x, no clamp mask) at depths up to 64; 4 elsewhere
    const bool async_path = p->epi.kind != FBCORR_EPI_CLAMP && p->D % 4 == 0 && p->N % 4 == 0;
    p->dw_tn = (p->dw_pk == 2 && async_path && p->D <= 64) ? 8 : 4;
    int tn_env = 0, ng_env = 0, qb_env = 0;   // FBCORR_DW_TILE="tn,ng,qb" (tile sweeps)
    if (sscanf(env_str("FBCORR_DW_TILE", "").c_str(), "%d,%d,%d", &tn_env, &ng_env, &qb_env) == 3 &&
        (tn_env == 4 || tn_env == 8) && ng_env >= 1 && ng_env * p->D <= 1024 && qb_env >= 8 && qb_env <= 256)
        p->dw_tn = tn_env;
    else
        ng_env = qb_env = 0;
    const long ngroups_needed = (p->N + p->dw_tn - 1) / p->dw_tn;
    p->dw_ng = (int)std::max(1L, std::min<long>((p->dw_tn == 8 ? 128 : 256) / std::max<int64_t>(1, p->D),
                                                ngroups_needed));
    p->dw_qb = 64;
    if (ng_env) {
        p->dw_ng = (int)std::min<long>(ng_env, ngroups_needed);
        p->dw_qb = qb_env;
    }
    p->dw_nblocks = (int)((p->N + (long)p->dw_tn * p->dw_ng - 1) / ((long)p->dw_tn * p->dw_ng));
    long want = (4L * std::max(1, p->dev.sm_count) + p->fh * p->dw_nblocks - 1) /
                (p->fh * p->dw_nblocks);
    want = std::max(1L, std::min<long>(want, std::min<long>(p->Ho, 256)));
    p->dw_rows_per_chunk = (int)((p->Ho + want - 1) / want);
    p->dw_chunks = (int)((p->Ho + p->dw_rows_per_chunk - 1) / p->dw_rows_per_chunk);
    p->ws_bwd = (size_t)p->dw_chunks * p->N * p->fh * p->fw * p->D * sizeof(float);
}

}  // namespace

fbcorr_status_t fbc::validate_shapes(const int64_t* in, const int64_t* fs, fbcorr_dtype_t dtype,
                                     const fbcorr_epilogue_t& epi) {
    if (!in || !fs) return set_error(FBCORR_ERR_INVALID_ARG, "null shape array");
    if (dtype != FBCORR_F32 && dtype != FBCORR_BF16 && dtype != FBCORR_BF16X3)
        return set_error(FBCORR_ERR_INVALID_ARG, "unknown dtype %d", (int)dtype);
    if (epi.kind != FBCORR_EPI_NONE && epi.kind != FBCORR_EPI_CLAMP && epi.kind != FBCORR_EPI_SNIPPET)
        return set_error(FBCORR_ERR_INVALID_ARG, "unknown epilogue kind %d", epi.kind);
    if (epi.kind == FBCORR_EPI_CLAMP && !(epi.lo <= epi.hi))
        return set_error(FBCORR_ERR_INVALID_ARG, "clamp needs lo <= hi (got %g, %g)", epi.lo, epi.hi);
    const int64_t H = in[0], W = in[1], D = in[2], N = fs[0], fh = fs[1], fw = fs[2], Dw = fs[3];
    if (H <= 0 || W <= 0 || D <= 0 || N <= 0 || fh <= 0 || fw <= 0 || Dw <= 0)
        return set_error(FBCORR_ERR_SHAPE, "every dimension must be positive");
    if (Dw != D) return set_error(FBCORR_ERR_SHAPE, "filter depth %lld != input depth %lld",
                                  (long long)Dw, (long long)D);
    if (fh > H || fw > W)
        return set_error(FBCORR_ERR_SHAPE, "filter %lldx%lld larger than input %lldx%lld",
                         (long long)fh, (long long)fw, (long long)H, (long long)W);
    const int64_t Ho = H - fh + 1, Wo = W - fw + 1;
    if (H > (1 << 20) || W > (1 << 20) || D > 4096 || N > 65535 || fh > 64 || fw > 64 ||
        H * W * D >= kMaxElems || Ho * Wo * N >= kMaxElems || N * fh * fw * D >= kMaxElems)
        return set_error(FBCORR_ERR_SHAPE, "shape exceeds the supported index range");
    return FBCORR_OK;
}

namespace {
}  // namespace

extern "C" {

}  // extern "C"

namespace {

// A snippet is kept a single C expression: no statements, blocks, directives or literals.
fbcorr_status_t validate_snippet(const char* expr) {
    if (!expr || !*expr) return set_error(FBCORR_ERR_INVALID_ARG, "empty snippet");
    const size_t n = strlen(expr);
    if (n > 1024) return set_error(FBCORR_ERR_INVALID_ARG, "snippet longer than 1024 characters");
    for (size_t i = 0; i < n; ++i) {
        const char c = expr[i];
        if (c == ';' || c == '{' || c == '}' || c == '#' || c == '"' || c == '\\' || c == '\'' ||
            (unsigned char)c < 0x20)
            return set_error(FBCORR_ERR_INVALID_ARG, "snippet must be one expression (character '%c' at %zu)",
                             c >= 0x20 ? c : '?', i);
    }
    return FBCORR_OK;
}

fbcorr_status_t plan_create(fbcorr_plan_t* out, const int64_t in_shape[3], const int64_t filt_shape[4],
                            fbcorr_dtype_t dtype, fbcorr_epilogue_t epilogue, const std::string& snippet) {
    *out = nullptr;
    FBC_TRY(validate_shapes(in_shape, filt_shape, dtype, epilogue));
    DeviceInfo dev;
    FBC_TRY(device_info(&dev));
    if (dev.cc_major != 10 || dev.cc_minor != 3)
        return set_error(FBCORR_ERR_UNSUPPORTED,
                         "libfbcorr is built for sm_103a (GB300); device %d is %s (cc %d.%d)",
                         dev.device, dev.name, dev.cc_major, dev.cc_minor);
    fbcorr_plan* p = new (std::nothrow) fbcorr_plan();
    if (!p) return set_error(FBCORR_ERR_OOM, "host allocation failed");
    p->H = in_shape[0];
    p->W = in_shape[1];
    p->D = in_shape[2];
    p->N = filt_shape[0];
    p->fh = filt_shape[1];
    p->fw = filt_shape[2];
    p->Ho = p->H - p->fh + 1;
    p->Wo = p->W - p->fw + 1;
    p->dtype = dtype;
    p->epi = epilogue;
    if (p->epi.kind == FBCORR_EPI_NONE) p->epi.lo = p->epi.hi = 0.f;
    p->snippet = snippet;
    p->dev = dev;

    fbcorr_status_t s = FBCORR_OK;
    if (cudaHostAlloc((void**)&p->err_host, sizeof(int), cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer((void**)&p->err_dev, p->err_host, 0) != cudaSuccess) {
        cudaGetLastError();
        s = set_error(FBCORR_ERR_OOM, "mapped host allocation for the error word failed");
    } else {
        *p->err_host = 0;
    }
    if (s == FBCORR_OK) {
        if (dtype == FBCORR_F32) {
            s = choose_fwd_f32(p);
        } else {
            p->fwd_kind = VarKind::Tensor;
            p->fwd_source = "fixed";
            s = tc_plan_create(&p->tc, (int)p->H, (int)p->W, (int)p->D, (int)p->N, (int)p->fh,
                               (int)p->fw, dtype == FBCORR_BF16X3 ? 1 : 0,
                               p->epi.kind == FBCORR_EPI_CLAMP ? 1 : 0, p->epi.lo, p->epi.hi, p->snippet, dev);
            if (s == FBCORR_OK) {
                p->ws_fwd = tc_workspace_bytes(p->tc);
                std::string spec = env_str("FBCORR_VARIANT", "");
                if ((spec.empty() || set_tc_spec(p, spec, "env") != FBCORR_OK) &&
                    (!tune_lookup(tune_key(p->dev, shape_key(p, "fwd")), &spec) ||
                     set_tc_spec(p, spec, "cache") != FBCORR_OK))
                    s = set_tc_heuristic(p);
                if (s == FBCORR_OK) clear_error();
            }
        }
    }
    if (s == FBCORR_OK) plan_dw_chunks(p);
    if (s != FBCORR_OK) {
        fbcorr_plan_destroy(p);
        return s;
    }
    const std::string at = env_str("FBCORR_AUTOTUNE", "0");
    if (at == "force" || (at == "1" && p->fwd_source == "heuristic")) {
        s = fbcorr_autotune(p, nullptr);
        if (s != FBCORR_OK) {
            fbcorr_plan_destroy(p);
            return s;
        }
    }
    logf("plan %lldx%lldx%lld * %lldx%lldx%lldx%lld dtype=%d: fwd=%s (%s)", (long long)p->H,
         (long long)p->W, (long long)p->D, (long long)p->N, (long long)p->fh, (long long)p->fw,
         (long long)p->D, (int)dtype, kind_name(p->fwd_kind), p->fwd_source.c_str());
    *out = p;
    return FBCORR_OK;
}

}  // namespace

extern "C" {

fbcorr_status_t fbcorr_plan_create(fbcorr_plan_t* out, const int64_t in_shape[3],
                                   const int64_t filt_shape[4], fbcorr_dtype_t dtype,
                                   fbcorr_epilogue_t epilogue) {
    clear_error();
    if (!out) return set_error(FBCORR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (epilogue.kind == FBCORR_EPI_SNIPPET)
        return set_error(FBCORR_ERR_INVALID_ARG, "a snippet epilogue needs fbcorr_plan_create_snippet");
    return plan_create(out, in_shape, filt_shape, dtype, epilogue, "");
}

fbcorr_status_t fbcorr_plan_create_snippet(fbcorr_plan_t* out, const int64_t in_shape[3],
                                           const int64_t filt_shape[4], fbcorr_dtype_t dtype,
                                           fbcorr_epilogue_t epilogue, const char* expr) {
    clear_error();
    if (!out) return set_error(FBCORR_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (epilogue.kind != FBCORR_EPI_SNIPPET)
        return set_error(FBCORR_ERR_INVALID_ARG, "epilogue.kind must be FBCORR_EPI_SNIPPET");
    FBC_TRY(validate_snippet(expr));
    return plan_create(out, in_shape, filt_shape, dtype, epilogue, expr);
}

fbcorr_status_t fbcorr_snippet_check(const int64_t in_shape[3], const int64_t filt_shape[4],
                                     fbcorr_dtype_t dtype, const char* expr, char* log, size_t cap) {
    clear_error();
    if (log && cap) log[0] = '\0';
    const fbcorr_epilogue_t epi{FBCORR_EPI_SNIPPET, 0.f, 0.f};
    FBC_TRY(validate_shapes(in_shape, filt_shape, dtype, epi));
    FBC_TRY(validate_snippet(expr));
    std::string lg;
    fbcorr_status_t st;
    fbcorr_plan tmp;
    tmp.H = in_shape[0]; tmp.W = in_shape[1]; tmp.D = in_shape[2];
    tmp.N = filt_shape[0]; tmp.fh = filt_shape[1]; tmp.fw = filt_shape[2];
    tmp.Ho = tmp.H - tmp.fh + 1; tmp.Wo = tmp.W - tmp.fw + 1;
    tmp.dtype = dtype;
    tmp.epi = epi;
    tmp.snippet = expr;
    const DirectProblem fp = fwd_problem(&tmp);
    if (dtype == FBCORR_F32) {
        const DirectTile t = direct_heuristic(fp, 200 * 1024, 148);
        st = rtcg_compile_only(direct_kernel_source(fp, t, kname_for("fbc_direct", fp, t)), &lg);
    } else {
        st = tc_snippet_check((int)in_shape[2], (int)filt_shape[2], dtype == FBCORR_BF16X3 ? 1 : 0, expr, &lg);
    }
    // and the kernel of rtcg_f32tc.cuh where the model prefers it
    F3Tile f3;
    if (st == FBCORR_OK && (dtype == FBCORR_F32 ? f3_wins(fp, 152, &f3) : f3_wins_bf16(fp, 152, plan_orders(&tmp), ~(size_t)0, &f3)))
        st = rtcg_compile_only(f3_kernel_source(fp, f3, f3_kernel_name(fp, f3)), &lg);
    if (st != FBCORR_OK && log && cap) snprintf(log, cap, "%s", lg.empty() ? fbcorr_last_error() : lg.c_str());
    return st;
}

fbcorr_status_t fbcorr_plan_profile(fbcorr_plan_t p, int capacity) {
    clear_error();
    if (!p || capacity < 0) return set_error(FBCORR_ERR_INVALID_ARG, "bad argument");
    for (auto e : p->prof_start) cudaEventDestroy(e);
    for (auto e : p->prof_stop) cudaEventDestroy(e);
    p->prof_start.clear();
    p->prof_stop.clear();
    p->prof_count = 0;
    for (int k = 0; k < capacity; ++k) {
        cudaEvent_t a, b;
        FBC_CUDA(cudaEventCreate(&a));
        if (cudaEventCreate(&b) != cudaSuccess) {
            cudaEventDestroy(a);
            return set_error(FBCORR_ERR_CUDA, "cudaEventCreate failed");
        }
        p->prof_start.push_back(a);
        p->prof_stop.push_back(b);
    }
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_profile_read(fbcorr_plan_t p, float* ms, int cap, int* n) {
    clear_error();
    if (!p || !n || (cap > 0 && !ms)) return set_error(FBCORR_ERR_INVALID_ARG, "bad argument");
    const int cnt = std::min(p->prof_count, cap);
    for (int k = 0; k < cnt; ++k) {
        FBC_CUDA(cudaEventSynchronize(p->prof_stop[k]));
        FBC_CUDA(cudaEventElapsedTime(&ms[k], p->prof_start[k], p->prof_stop[k]));
    }
    *n = cnt;
    p->prof_count = 0;
    return FBCORR_OK;
}

int plan_launches_per_forward(const fbcorr_plan* p) {
    return p->fwd_kind == VarKind::Tensor ? tc_launches(p->tc) : p->fwd_kind == VarKind::F32tc ? 2 : 1;
}

fbcorr_status_t fbcorr_plan_destroy(fbcorr_plan_t p) {
    clear_error();
    if (!p) return FBCORR_OK;
    for (auto e : p->prof_start) cudaEventDestroy(e);
    for (auto e : p->prof_stop) cudaEventDestroy(e);
    hostpipe_destroy(p->hostpipe);
    if (p->bwd_side) cudaStreamDestroy(p->bwd_side);
    if (p->bwd_fork) cudaEventDestroy(p->bwd_fork);
    if (p->bwd_join) cudaEventDestroy(p->bwd_join);
    if (p->tc) tc_plan_destroy(p->tc);
    if (p->err_host) cudaFreeHost(p->err_host);
    delete p;
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_out_shape(fbcorr_plan_t p, int64_t out[3]) {
    clear_error();
    if (!p || !out) return set_error(FBCORR_ERR_INVALID_ARG, "NULL argument");
    out[0] = p->Ho;
    out[1] = p->Wo;
    out[2] = p->N;
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_workspace_size(fbcorr_plan_t p, size_t* fwd, size_t* bwd) {
    clear_error();
    if (!p) return set_error(FBCORR_ERR_INVALID_ARG, "NULL plan");
    if (fwd) *fwd = p->ws_fwd;
    if (bwd) *bwd = p->ws_bwd;
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_scratch_size(fbcorr_plan_t p, size_t* fwd, size_t* bwd) {
    clear_error();
    if (!p) return set_error(FBCORR_ERR_INVALID_ARG, "NULL plan");
    if (fwd) *fwd = p->fwd_kind == VarKind::F32tc ? p->fwd_f3.ws_bytes : p->ws_fwd;
    if (bwd) {
        *bwd = p->ws_bwd;
        if (p->epi.kind != FBCORR_EPI_SNIPPET) {
            FBC_TRY(prepare_backward(p));
            if (p->dx_kind == VarKind::F32tc) *bwd = dx_scratch_offset(p) + p->dx_f3.ws_bytes;
            if (p->dw_f3.parts) *bwd = dw_scratch_offset(p) + p->dw_f3.ws_bytes;
        }
    }
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_forward(fbcorr_plan_t p, const float* x, const float* w, float* y, void* ws,
                               size_t ws_bytes, fbcorr_stream_t stream) {
    clear_error();
    if (!p || !x || !w || !y) return set_error(FBCORR_ERR_INVALID_ARG, "NULL argument");
    if (!aligned16(x) || !aligned16(w) || !aligned16(y))
        return set_error(FBCORR_ERR_ALIGNMENT, "x, w and y must be 16-byte aligned");
    if (p->ws_fwd > 0 && (!ws || ws_bytes < p->ws_fwd || !aligned16(ws)))
        return set_error(FBCORR_ERR_WORKSPACE, "forward needs %zu bytes of aligned workspace (got %zu)",
                         p->ws_fwd, ws ? ws_bytes : (size_t)0);
    cudaStream_t s = (cudaStream_t)stream;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (p->prof_count < (int)p->prof_start.size()) {
        e0 = p->prof_start[p->prof_count];
        e1 = p->prof_stop[p->prof_count];
        ++p->prof_count;
    }
    fbcorr_status_t st = FBCORR_OK;
    switch (p->fwd_kind) {
        case VarKind::Direct:
            if (e0) FBC_CUDA(cudaEventRecord(e0, s));
            st = run_direct(p->fwd_kernel, fwd_problem(p), p->fwd_tile, x, nullptr, w, y,
                            p->epi.lo, p->epi.hi, s);
            if (e1 && st == FBCORR_OK) FBC_CUDA(cudaEventRecord(e1, s));
            return st;
        case VarKind::Default:
            if (e0) FBC_CUDA(cudaEventRecord(e0, s));
            st = run_default(fwd_problem(p), x, nullptr, w, y, p->epi.lo, p->epi.hi, s);
            if (e1 && st == FBCORR_OK) FBC_CUDA(cudaEventRecord(e1, s));
            return st;
        case VarKind::F32tc:
            if (e0) FBC_CUDA(cudaEventRecord(e0, s));
            st = ws && aligned16(ws) && ws_bytes >= p->fwd_f3.ws_bytes
                     ? f3_run(p->fwd_f3, fwd_problem(p), x, nullptr, w, y, ws, p->epi.lo, p->epi.hi, p->err_dev, s)
                     : run_fma(p->fwd_kernel, p->fwd_tile, fwd_problem(p), x, nullptr, w, y, p->epi.lo, p->epi.hi, s);
            if (e1 && st == FBCORR_OK) FBC_CUDA(cudaEventRecord(e1, s));
            return st;
        case VarKind::Tensor:
            if (p->tc_packed) {
                if (e0) FBC_CUDA(cudaEventRecord(e0, s));
                st = f3_run(p->fwd_f3, fwd_problem(p), x, nullptr, w, y, ws, p->epi.lo, p->epi.hi, p->err_dev, s);
                if (e1 && st == FBCORR_OK) FBC_CUDA(cudaEventRecord(e1, s));
                return st;
            }
            return tc_forward(p->tc, x, w, y, ws, p->err_dev, s, e0, e1);
    }
    return set_error(FBCORR_ERR_INTERNAL, "bad variant kind");
}

fbcorr_status_t fbcorr_backward(fbcorr_plan_t p, const float* x, const float* w, const float* g,
                                const float* y, float* dx, float* dw, void* ws, size_t ws_bytes,
                                fbcorr_stream_t stream) {
    clear_error();
    if (!p || !g) return set_error(FBCORR_ERR_INVALID_ARG, "NULL plan or gradient");
    if (p->epi.kind == FBCORR_EPI_SNIPPET)
        return set_error(FBCORR_ERR_UNSUPPORTED, "a snippet epilogue is forward-only (no derivative)");
    if (dw && !x) return set_error(FBCORR_ERR_INVALID_ARG, "dw needs x");
    if (dx && !w) return set_error(FBCORR_ERR_INVALID_ARG, "dx needs w");
    const bool clamp = p->epi.kind == FBCORR_EPI_CLAMP;
    if (clamp && !y) return set_error(FBCORR_ERR_INVALID_ARG, "a clamp epilogue needs y for its mask");
    const void* ptrs[] = {x, w, g, clamp ? y : nullptr, dx, dw};
    for (const void* q : ptrs)
        if (q && !aligned16(q)) return set_error(FBCORR_ERR_ALIGNMENT, "tensors must be 16-byte aligned");
    if (!dx && !dw) return FBCORR_OK;
    if (dw && (!ws || ws_bytes < p->ws_bwd || !aligned16(ws)))
        return set_error(FBCORR_ERR_WORKSPACE, "backward needs %zu bytes of aligned workspace (got %zu)",
                         p->ws_bwd, ws ? ws_bytes : (size_t)0);
    FBC_TRY(prepare_backward(p));
    cudaStream_t s = (cudaStream_t)stream;
    const float* m = clamp ? y : nullptr;
    // both gradients: dL/dw on the side stream, forked after the work already on
    // `s` and joined back before anything queued on `s` after this call, so the two
    // gradients' kernels fill each other's idle SMs.  Not when both run on the tensor
    // cores: each fills every SM, and the fork costs the host four event calls
    // (autograd step 256x256x16 * 64x7x7, bound by the host: 261 to 207 us together
    // with the lighter Python calls)
    const bool f3_dx = dx && p->dx_kind == VarKind::F32tc && ws && aligned16(ws) &&
                       ws_bytes >= dx_scratch_offset(p) + p->dx_f3.ws_bytes;
    const bool f3_dw = dw && p->dw_f3.parts && ws_bytes >= dw_scratch_offset(p) + p->dw_f3.ws_bytes;
    const bool fork = dx && dw && p->bwd_side && !(f3_dx && f3_dw);
    cudaStream_t sw = fork ? p->bwd_side : s;
    if (fork) {
        FBC_CUDA(cudaEventRecord(p->bwd_fork, s));
        FBC_CUDA(cudaStreamWaitEvent(sw, p->bwd_fork, 0));
    }
    if (dw) {
        float* part = (float*)ws;
        // with scratch: the tensor-core kernel; the FMA kernel behind it then runs only
        // for inputs that it flags (non-finite or tiny values)
        const float* part3 = nullptr;
        const int* flags = nullptr;
        if (f3_dw)
            FBC_TRY(f3dw_run(p->dw_f3, dw_problem(p), x, g, m ? m : g, (uint8_t*)ws + dw_scratch_offset(p), p->epi.lo,
                             p->epi.hi, p->err_dev, &part3, &flags, sw));
        if (p->dw_kind == VarKind::Direct) {
            DwArgsK a{x, g, m ? m : g, part, (int)p->H, (int)p->W, (int)p->Ho, (int)p->Wo, (int)p->N,
                      p->dw_rows_per_chunk, p->epi.lo, p->epi.hi, flags, p->dw_f3.grid};
            void* args[] = {&a};
            dim3 grid((unsigned)p->dw_chunks, (unsigned)p->fh, (unsigned)p->dw_nblocks);
            FBC_TRY(launch(p->dw_kernel, grid, args, sw));
        } else {
            FBC_CUDA(launch_default_dw(x, g, m ? m : g, part, (int)p->H, (int)p->W, (int)p->D,
                                       (int)p->Ho, (int)p->Wo, (int)p->N, (int)p->fh, (int)p->fw,
                                       p->dw_chunks, p->dw_rows_per_chunk, clamp ? 1 : 0, p->epi.lo,
                                       p->epi.hi, sw));
        }
        const long long elems = (long long)p->N * p->fh * p->fw * p->D;
        FBC_CUDA(part3 ? launch_dw_reduce(part3, dw, p->dw_f3.parts, elems, sw, flags, p->dw_f3.grid, part, p->dw_chunks)
                       : launch_dw_reduce(part, dw, p->dw_chunks, elems, sw));
    }
    if (fork) FBC_CUDA(cudaEventRecord(p->bwd_join, sw));
    fbcorr_status_t st = FBCORR_OK;
    if (dx) {
        const DirectProblem pr = dx_problem(p);
        st = f3_dx ? f3_run(p->dx_f3, pr, g, m, w, dx, (uint8_t*)ws + dx_scratch_offset(p), p->epi.lo, p->epi.hi,
                            p->err_dev, s)
             : p->dx_kind != VarKind::Default
                 ? run_fma(p->dx_kernel, p->dx_tile, pr, g, m, w, dx, p->epi.lo, p->epi.hi, s)
                 : run_default(pr, g, m, w, dx, p->epi.lo, p->epi.hi, s);
    }
    // the join even when dL/dx failed to launch: nothing on `s` may overtake dL/dw
    if (fork) FBC_CUDA(cudaStreamWaitEvent(s, p->bwd_join, 0));
    return st;
}

fbcorr_status_t fbcorr_plan_set_variant(fbcorr_plan_t p, const char* spec) {
    clear_error();
    if (!p || !spec) return set_error(FBCORR_ERR_INVALID_ARG, "NULL argument");
    const std::string s = spec;
    if (p->dtype != FBCORR_F32) {
        if (s == "tuned") return fbcorr_autotune(p, nullptr);
        if (s != "heuristic") return set_tc_spec(p, s, "forced");
        FBC_TRY(tc_set_spec(p->tc, tc_candidates(p->tc).front()));
        return set_tc_heuristic(p);
    }
    if (s == "heuristic") return set_fwd_spec(p, heuristic_spec(fwd_problem(p), p->dev), "heuristic");
    if (s == "tuned") return fbcorr_autotune(p, nullptr);
    return set_fwd_spec(p, s, "forced");
}

static fbcorr_status_t autotune_tc(fbcorr_plan_t p, fbcorr_stream_t stream);

static fbcorr_status_t tune_direct(fbcorr_plan_t p, const DirectProblem& pr, cudaStream_t s,
                                   const char* what, std::string* best_spec, float* best_ms_out) {
    int topk = atoi(env_str("FBCORR_TUNE_TOPK", "48").c_str());
    return tune_direct_problem(p->dev, pr, s, 0, 64, smem_limit(p->dev), std::max(1, topk), p->snippet.empty(),
                               what, best_spec, best_ms_out);
}

fbcorr_status_t fbcorr_autotune(fbcorr_plan_t p, fbcorr_stream_t stream) {
    clear_error();
    if (!p) return set_error(FBCORR_ERR_INVALID_ARG, "NULL plan");
    cudaStream_t s = (cudaStream_t)stream;
    if (p->dtype != FBCORR_F32) return autotune_tc(p, stream);
    // forward
    std::string best;
    float ms = 0.f;
    FBC_TRY(tune_direct(p, fwd_problem(p), s, "fwd", &best, &ms));
    float f3_ms = 0.f;
    std::string f3;
    FBC_TRY(f3_tune(p->dev, fwd_problem(p), s, p->err_dev, &f3_ms, &f3));
    // the fastest FMA kernel is kept as well, for calls without scratch
    const std::string fma = best;
    tune_store(tune_key(p->dev, shape_key(p, "fwd") + "|fma"), fma);
    if (!f3.empty() && f3_ms < ms) {
        best = f3;
        ms = f3_ms;
    }
    FBC_TRY(set_fwd_spec(p, best, "tuned", fma));
    tune_store(tune_key(p->dev, shape_key(p, "fwd")), best);
    logf("autotune fwd picked %s (%.4f ms)", best.c_str(), ms);
    // dL/dx: the same generated kernel family on the flipped problem
    std::string best_dx;
    FBC_TRY(tune_direct(p, dx_problem(p), s, "dx", &best_dx, &ms));
    FBC_TRY(f3_tune(p->dev, dx_problem(p), s, p->err_dev, &f3_ms, &f3));
    tune_store(tune_key(p->dev, shape_key(p, "dx") + "|fma"), best_dx);
    if (!f3.empty() && f3_ms < ms) {
        best_dx = f3;
        ms = f3_ms;
    }
    tune_store(tune_key(p->dev, shape_key(p, "dx")), best_dx);
    logf("autotune dx picked %s (%.4f ms)", best_dx.c_str(), ms);
    p->bwd_ready = false;   // rebuilt from the cache entry on the next backward call
    return FBCORR_OK;
}

}  // extern "C"

// Values in [-scale, scale) from an integer hash of the index (the "lowbias32"
// mixer of C. Wellons' hash-prospector), for timing runs only.
__global__ void fbc_fill_pattern(float* p, size_t n, float scale, unsigned seed) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        unsigned h = (unsigned)i ^ seed;
        h ^= h >> 16;
        h *= 0x7feb352du;
        h ^= h >> 15;
        h *= 0x846ca68bu;
        h ^= h >> 16;
        p[i] = scale * ((float)(h >> 8) * (2.0f / 16777216.0f) - 1.0f);
    }
}

cudaError_t fbc::launch_fill_pattern(float* p, size_t n, float scale, unsigned seed, cudaStream_t s) {
    fbc_fill_pattern<<<256, 256, 0, s>>>(p, n, scale, seed);
    return cudaGetLastError();
}

extern "C" {

// Time every feasible tensor-core configuration (ring depths, filter-tile
// width) and keep the fastest -- the same measured grid search as for the
// generated FP32 kernels.
static fbcorr_status_t autotune_tc(fbcorr_plan_t p, fbcorr_stream_t stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const std::vector<std::string> specs = tc_candidates(p->tc);
    const std::string old = tc_spec(p->tc);
    const bool packed_before = p->tc_packed;
    float *x = nullptr, *w = nullptr, *y = nullptr;
    void* ws = nullptr;
    const size_t xb = (size_t)p->H * p->W * p->D * 4, wb = (size_t)p->N * p->fh * p->fw * p->D * 4,
                 yb = (size_t)p->Ho * p->Wo * p->N * 4;
    if (cudaMalloc(&x, xb) != cudaSuccess || cudaMalloc(&w, wb) != cudaSuccess ||
        cudaMalloc(&y, yb) != cudaSuccess || cudaMalloc(&ws, p->ws_fwd) != cudaSuccess) {
        cudaFree(x); cudaFree(w); cudaFree(y); cudaFree(ws);
        cudaGetLastError();
        return set_error(FBCORR_ERR_OOM, "autotune buffers");
    }
    p->tc_packed = false;   // the candidates below are the plan's own kernel
    // non-zero operands: the tensor cores draw (and the clocks follow) more power
    // on real data than on zeros, so timings on zeros would favour the wrong spec
    launch_fill_pattern(x, xb / 4, 1.0f, 0x1234u, s);
    launch_fill_pattern(w, wb / 4, 0.05f, 0x5678u, s);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    std::string best;
    float best_ms = 1e30f;
    fbcorr_status_t status = FBCORR_OK;
    std::vector<std::pair<float, std::string>> timed;   // (median single-step ms, spec)
    tc_precompile(p->tc, specs);   // the generated kernels of all candidates, on host threads
    for (const auto& sp : specs) {
        if (tc_set_spec(p->tc, sp) != FBCORR_OK) continue;
        std::vector<float> ms;
        bool ok = true;
        for (int r = 0; r < 2 && ok; ++r) ok = fbcorr_forward(p, x, w, y, ws, p->ws_fwd, stream) == FBCORR_OK;
        for (int r = 0; r < 5 && ok; ++r) {
            cudaEventRecord(e0, s);
            ok = fbcorr_forward(p, x, w, y, ws, p->ws_fwd, stream) == FBCORR_OK;
            cudaEventRecord(e1, s);
            if (cudaEventSynchronize(e1) != cudaSuccess) ok = false;
            float t = 0.f;
            cudaEventElapsedTime(&t, e0, e1);
            ms.push_back(t);
        }
        if (!ok || fbcorr_plan_device_status(p, 0) != FBCORR_OK) {
            status = set_error(FBCORR_ERR_CUDA, "autotune run of %s failed", sp.c_str());
            break;
        }
        std::sort(ms.begin(), ms.end());
        logf("autotune %s: %.4f ms", sp.c_str(), ms[ms.size() / 2]);
        timed.push_back({ms[ms.size() / 2], sp});
    }
    // Finalists: single steps separate candidates within about 1 %, and the clock
    // drifts as the GPU warms up over the sweep, so the six fastest are timed
    // again, round-robin over three rounds, as runs of 20 back-to-back steps
    // (the way the forward is used); the best round of each decides.
    if (status == FBCORR_OK && !timed.empty()) {
        std::sort(timed.begin(), timed.end());
        const size_t nf = std::min<size_t>(timed.size(), 6);
        std::vector<float> fin(nf, 1e30f);
        for (int round = 0; round < 3 && status == FBCORR_OK; ++round)
            for (size_t f = 0; f < nf && status == FBCORR_OK; ++f) {
                if (tc_set_spec(p->tc, timed[f].second) != FBCORR_OK) continue;
                bool ok = fbcorr_forward(p, x, w, y, ws, p->ws_fwd, stream) == FBCORR_OK;
                cudaEventRecord(e0, s);
                for (int r = 0; r < 20 && ok; ++r) ok = fbcorr_forward(p, x, w, y, ws, p->ws_fwd, stream) == FBCORR_OK;
                cudaEventRecord(e1, s);
                if (!ok || cudaEventSynchronize(e1) != cudaSuccess || fbcorr_plan_device_status(p, 0) != FBCORR_OK) {
                    status = set_error(FBCORR_ERR_CUDA, "autotune run of %s failed", timed[f].second.c_str());
                    break;
                }
                float t = 0.f;
                cudaEventElapsedTime(&t, e0, e1);
                fin[f] = std::min(fin[f], t / 20.f);
            }
        for (size_t f = 0; f < nf; ++f) {
            logf("autotune finalist %s: %.4f ms", timed[f].second.c_str(), fin[f]);
            if (fin[f] < best_ms) {
                best_ms = fin[f];
                best = timed[f].second;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(x); cudaFree(w); cudaFree(y); cudaFree(ws);
    if (status != FBCORR_OK || best.empty()) {
        tc_set_spec(p->tc, old);
        p->tc_packed = packed_before;
        return status != FBCORR_OK ? status : set_error(FBCORR_ERR_INTERNAL, "no variant ran");
    }
    FBC_TRY(set_tc_spec(p, best, "tuned"));
    float packed_ms = 0.f;
    std::string packed;
    FBC_TRY(f3_tune(p->dev, fwd_problem(p), s, p->err_dev, &packed_ms, &packed, plan_orders(p), p->ws_fwd));
    if (!packed.empty() && packed_ms < best_ms && set_tc_spec(p, packed, "tuned") == FBCORR_OK) {
        best = packed;
        best_ms = packed_ms;
    }
    tune_store(tune_key(p->dev, shape_key(p, "fwd")), best);
    logf("autotune picked %s (%.4f ms)", best.c_str(), best_ms);
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_info(fbcorr_plan_t p, char* buf, size_t cap) {
    clear_error();
    if (!p || !buf || cap == 0) return set_error(FBCORR_ERR_INVALID_ARG, "NULL argument");
    std::ostringstream o;
    o << "{\"in\":[" << p->H << "," << p->W << "," << p->D << "],\"filt\":[" << p->N << "," << p->fh
      << "," << p->fw << "," << p->D << "],\"out\":[" << p->Ho << "," << p->Wo << "," << p->N
      << "],\"dtype\":" << (int)p->dtype << ",\"epilogue\":" << p->epi.kind << ",\"fwd\":{\"kind\":\""
      << kind_name(p->fwd_kind) << "\",\"source\":\"" << p->fwd_source << "\"";
    if (p->fwd_kind == VarKind::Direct) {
        o << ",\"spec\":\"" << direct_tile_spec(p->fwd_tile) << "\",\"smem\":" << p->fwd_kernel.smem
          << ",\"threads\":" << p->fwd_kernel.threads << ",\"kernel\":\"" << p->fwd_kernel.name
          << "\",\"source_hash\":\"" << hex64(p->fwd_kernel.src_hash) << "\"";
    } else if (p->fwd_kind == VarKind::F32tc) {
        o << ",\"spec\":\"" << f3_spec(p->fwd_f3.tile) << "\",\"smem\":" << p->fwd_f3.kernel.smem << ",\"threads\":"
          << p->fwd_f3.kernel.threads << ",\"grid\":" << p->fwd_f3.grid << ",\"slots\":[" << p->fwd_f3.na << ","
          << p->fwd_f3.nb << "],\"kernel\":\"" << p->fwd_f3.kernel.name << "\",\"source_hash\":\""
          << hex64(p->fwd_f3.kernel.src_hash) << "\",\"fma\":\""
          << (p->fwd_kernel.fn ? direct_tile_spec(p->fwd_tile) : "default") << "\"";
    } else if (p->fwd_kind == VarKind::Default) {
        o << ",\"spec\":\"default\"";
    } else if (p->tc_packed) {
        o << ",\"spec\":\"" << f3_spec(p->fwd_f3.tile) << "\",\"detail\":{\"precision\":\""
          << (p->dtype == FBCORR_BF16X3 ? "bf16x3" : "bf16") << "\",\"filter_tiles\":" << p->fwd_f3.filter_tiles
          << ",\"tail_half_tiles\":0,\"smem\":" << p->fwd_f3.kernel.smem << ",\"grid\":" << p->fwd_f3.grid
          << ",\"threads\":" << p->fwd_f3.kernel.threads << ",\"kernel\":\"" << p->fwd_f3.kernel.name
          << "\",\"source_hash\":\"" << hex64(p->fwd_f3.kernel.src_hash) << "\"}";
    } else if (p->tc) {
        o << ",\"spec\":\"" << tc_spec(p->tc) << "\",\"detail\":" << tc_describe(p->tc);
    }
    o << ",\"launches\":" << plan_launches_per_forward(p) << "},\"bwd_ready\":" << (p->bwd_ready ? 1 : 0);
    if (p->bwd_ready) {
        o << ",\"dx\":{\"kind\":\"" << kind_name(p->dx_kind) << "\"";
        if (p->dx_kind == VarKind::Direct) o << ",\"spec\":\"" << direct_tile_spec(p->dx_tile) << "\"";
        if (p->dx_kind == VarKind::F32tc)
            o << ",\"spec\":\"" << f3_spec(p->dx_f3.tile) << "\",\"fma\":\""
              << (p->dx_kernel.fn ? direct_tile_spec(p->dx_tile) : "default") << "\"";
        o << "},\"dw\":{\"kind\":\"" << kind_name(p->dw_kind) << "\",\"threads\":" << p->D * p->dw_ng
          << ",\"filters_per_cta\":" << p->dw_tn * p->dw_ng << ",\"packed_pairs\":" << p->dw_pk << ",\"min_blocks\":" << p->dw_mb
          << ",\"registers\":" << p->dw_regs << ",\"tile\":[" << p->dw_tn << "," << p->dw_ng << "," << p->dw_qb << "]"
          << ",\"chunks\":" << p->dw_chunks
          << ",\"rows_per_chunk\":" << p->dw_rows_per_chunk;
        if (p->dw_f3.parts)
            o << ",\"f32tc\":{\"kernel\":\"" << p->dw_f3.kernel.name << "\",\"grid\":" << p->dw_f3.grid
              << ",\"splits\":" << p->dw_f3.tile.splits << "}";
        o << "}";
    }
    o << ",\"ws_fwd\":" << p->ws_fwd << ",\"ws_bwd\":" << p->ws_bwd << ",\"sm_count\":"
      << p->dev.sm_count << "}";
    const std::string s = o.str();
    snprintf(buf, cap, "%s", s.c_str());
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_candidates(fbcorr_plan_t p, char* buf, size_t cap) {
    clear_error();
    if (!p || !buf || cap == 0) return set_error(FBCORR_ERR_INVALID_ARG, "NULL argument");
    std::vector<std::string> specs;
    if (p->dtype == FBCORR_F32) {
        const int topk = std::max(1, atoi(env_str("FBCORR_TUNE_TOPK", "48").c_str()));
        specs = direct_tuning_specs(direct_ranked(fwd_problem(p), smem_limit(p->dev), p->dev.sm_count, 0, 64),
                                    topk, (int)p->D);
        if (p->snippet.empty()) specs.push_back("default");
    } else {
        specs = tc_candidates(p->tc);
    }
    for (const F3Tile& t : f3_candidates(fwd_problem(p), p->dev.sm_count, plan_orders(p),
                                         p->dtype == FBCORR_F32 ? ~(size_t)0 : p->ws_fwd))
        specs.push_back(f3_spec(t));
    std::string s;
    for (const auto& sp : specs) s += sp + "\n";
    if (s.size() + 1 > cap) return set_error(FBCORR_ERR_INVALID_ARG, "buffer too small (%zu bytes needed)", s.size() + 1);
    memcpy(buf, s.c_str(), s.size() + 1);
    return FBCORR_OK;
}

fbcorr_status_t fbcorr_plan_device_status(fbcorr_plan_t p, int clear) {
    clear_error();
    if (!p) return set_error(FBCORR_ERR_INVALID_ARG, "NULL plan");
    const int v = p->err_host ? *(volatile int*)p->err_host : 0;
    if (clear && p->err_host) *(volatile int*)p->err_host = 0;
    const fbcorr_status_t bands = hostpipe_device_status(p->hostpipe, clear);
    if (v != 0) return set_error(FBCORR_ERR_TIMEOUT, "a kernel gave up a bounded wait (code %d)", v);
    if (bands != FBCORR_OK) return set_error(FBCORR_ERR_TIMEOUT, "a band kernel of fbcorr_forward_host gave up a bounded wait");
    return FBCORR_OK;
}

const char* fbcorr_status_string(fbcorr_status_t s) {
    switch (s) {
        case FBCORR_OK: return "FBCORR_OK";
        case FBCORR_ERR_INVALID_ARG: return "FBCORR_ERR_INVALID_ARG";
        case FBCORR_ERR_SHAPE: return "FBCORR_ERR_SHAPE";
        case FBCORR_ERR_UNSUPPORTED: return "FBCORR_ERR_UNSUPPORTED";
        case FBCORR_ERR_ALIGNMENT: return "FBCORR_ERR_ALIGNMENT";
        case FBCORR_ERR_WORKSPACE: return "FBCORR_ERR_WORKSPACE";
        case FBCORR_ERR_CUDA: return "FBCORR_ERR_CUDA";
        case FBCORR_ERR_NVRTC: return "FBCORR_ERR_NVRTC";
        case FBCORR_ERR_OOM: return "FBCORR_ERR_OOM";
        case FBCORR_ERR_TIMEOUT: return "FBCORR_ERR_TIMEOUT";
        case FBCORR_ERR_INTERNAL: return "FBCORR_ERR_INTERNAL";
    }
    return "FBCORR_ERR_UNKNOWN";
}

const char* fbcorr_last_error(void) { return last_error_message(); }

const char* fbcorr_version(void) { return "fbcorr 0.1 sm_103a"; }

fbcorr_status_t fbcorr_rtcg_check(const int64_t in_shape[3], const int64_t filt_shape[4],
                                  fbcorr_epilogue_t epilogue, const char* spec, char* log,
                                  size_t cap) {
    clear_error();
    if (log && cap) log[0] = '\0';
    FBC_TRY(validate_shapes(in_shape, filt_shape, FBCORR_F32, epilogue));
    if (epilogue.kind == FBCORR_EPI_SNIPPET)
        return set_error(FBCORR_ERR_INVALID_ARG, "snippet epilogues are checked by fbcorr_snippet_check");
    fbcorr_plan tmp;
    tmp.H = in_shape[0];
    tmp.W = in_shape[1];
    tmp.D = in_shape[2];
    tmp.N = filt_shape[0];
    tmp.fh = filt_shape[1];
    tmp.fw = filt_shape[2];
    tmp.Ho = tmp.H - tmp.fh + 1;
    tmp.Wo = tmp.W - tmp.fw + 1;
    tmp.epi = epilogue;
    const std::string sp = spec ? spec : "heuristic";
    if (sp.compare(0, 8, "tcgen05:") == 0) {
        // the generated tensor-core kernel of this spec, BF16 and split BF16
        std::string lg;
        const fbcorr_status_t st = tc_rtcg_check((int)tmp.D, (int)tmp.fw, sp, &lg);
        if (st != FBCORR_OK && log && cap) snprintf(log, cap, "%s", lg.empty() ? fbcorr_last_error() : lg.c_str());
        return st;
    }
    const size_t lim = 200 * 1024;
    const DirectProblem fp = fwd_problem(&tmp), bp = dx_problem(&tmp);
    F3Tile f3;
    if (f3_parse_spec(sp, &f3) || sp == "f32tc") {
        // the FP32 tensor-core kernels of the forward (this tile, or the heuristic's), of
        // dL/dx, and of dL/dw where a plan runs it
        for (const DirectProblem* pr : {&fp, &bp}) {
            const std::vector<F3Tile> ranked = f3_ranked(*pr, 152, nullptr);
            if (ranked.empty())
                return set_error(FBCORR_ERR_UNSUPPORTED, "the FP32 tensor-core kernel does not take this shape");
            const F3Tile ft = pr == &fp && sp != "f32tc" ? f3 : ranked.front();
            if (f3_ws_bytes(*pr, ft) == 0)     // before anything is derived from the tile
                return set_error(FBCORR_ERR_UNSUPPORTED, "variant %s does not fit this shape", f3_spec(ft).c_str());
            std::string lg;
            const fbcorr_status_t st = rtcg_compile_only(f3_kernel_source(*pr, ft, f3_kernel_name(*pr, ft)), &lg);
            if (st != FBCORR_OK) {
                if (log && cap) snprintf(log, cap, "%s", lg.c_str());
                return st;
            }
        }
        F3DwTile dt;
        if (!f3dw_wins(dw_problem(&tmp), 152, &dt)) return FBCORR_OK;
        std::string name, lg;
        const fbcorr_status_t st = rtcg_compile_only(f3dw_kernel_source(dw_problem(&tmp), dt, &name), &lg);
        if (st != FBCORR_OK && log && cap) snprintf(log, cap, "%s", lg.c_str());
        return st;
    }
    DirectTile t;
    if (sp == "heuristic")
        t = direct_heuristic(fp, lim, 148);
    else if (!parse_direct_spec(sp, &t))
        return set_error(FBCORR_ERR_INVALID_ARG, "unknown variant spec '%s'", sp.c_str());
    DirectTile tb = direct_heuristic(bp, lim, 148);
    if (t.ks_chunked()) {
        // a chunked K-split spec is a dL/dx tile: checked on the flipped problem
        if (!ks_chunked_fits(bp))
            return set_error(FBCORR_ERR_UNSUPPORTED, "spec '%s' is a dL/dx tile that this shape does not take",
                             sp.c_str());
        tb = t;
        t = direct_heuristic(fp, lim, 148);
    }
    const int mask = epilogue.kind == FBCORR_EPI_CLAMP ? 1 : 0;
    const std::string srcs[3] = {
        direct_kernel_source(fp, t, kname_for("fbc_direct", fp, t)),
        direct_kernel_source(bp, tb, kname_for("fbc_direct", bp, tb)),
        dw_kernel_source((int)tmp.fh, (int)tmp.fw, (int)tmp.D, 4,
                         (int)std::max<int64_t>(1, std::min<int64_t>(256 / tmp.D, (tmp.N + 3) / 4)), 64,
                         mask, 2, "fbc_dw_check", 3)};
    for (const auto& src : srcs) {
        std::string lg;
        fbcorr_status_t s = rtcg_compile_only(src, &lg);
        if (s != FBCORR_OK) {
            if (log && cap) snprintf(log, cap, "%s", lg.c_str());
            return s;
        }
    }
    return FBCORR_OK;
}

}  // extern "C"

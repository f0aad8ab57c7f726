// f32tc_kernel.cu -- host side of the FP32 tensor-core correlation (rtcg_f32tc.cuh):
// tile selection, shared-memory layout, run-time generation and launch.  Two launches
// per call (the split of the bank, and the correlation as its programmatic
// dependent); the forward and dL/dx are both DirectProblems.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <sstream>
#include <utility>

#include "f32tc_params.h"
#include "internal.h"

namespace fbc {

namespace {

constexpr size_t kSmemMax = 227 * 1024 - 1024;   // leave room for static shared memory
constexpr int kBarBytes = 512;

// The kernel template's derived constants (FbcF3Cfg of rtcg_f32tc.cuh).
struct Geometry {
    int pp, pl, s, ncg, ntg, rows, nu, ls, ka;
    size_t aslot, bstage, bunit;
    long long bank_chunks;   // per filter tile
};

Geometry geometry(const DirectProblem& pr, const F3Tile& t) {
    Geometry g;
    const bool pack = t.gc == 8;
    g.pp = !pack ? 1 : pr.c <= 1 ? 8 : pr.c <= 2 ? 4 : pr.c <= 4 ? 2 : 1;
    g.pl = pack ? 1 : t.gc / 8;
    g.s = pack ? (t.jt + 2 * g.pp - 1) / (2 * g.pp) : t.jt * (t.gc / 16);
    g.ncg = (pr.c + t.gc - 1) / t.gc;
    g.ntg = (pr.fw + t.jt - 1) / t.jt;
    g.rows = pr.fh + t.r - 1;
    g.nu = (g.rows + t.ru - 1) / t.ru * g.ncg * g.ntg;
    g.ls = pack ? 128 + (2 * g.s - 1) * g.pp : 128 + t.jt - 1;
    const int lp = g.pl == 4 ? (g.ls + 5) / 8 * 8 + 2 : g.pl == 2 ? (g.ls + 3) / 8 * 8 + 4 : g.ls;
    g.aslot = ((size_t)t.ru * t.ord * g.pl * lp * 16 + 127) / 128 * 128;
    g.bstage = (size_t)(t.ord * t.nt >= 144 ? 2 : t.ord * t.nt >= 96 ? 4 : 8) * 32 * t.ord * t.nt;
    g.bunit = (size_t)t.ru * g.s * 32 * t.ord * t.nt;
    const bool va = pr.c % 4 == 0;
    const int items = t.ru * (va && g.pp == 2 ? g.ls + 1 : g.ls) * (!va ? g.pl : g.pp == 2 ? 1 : t.gc / 4);
    g.ka = (items + 32 * FBC_F3_CONV_WARPS - 1) / (32 * FBC_F3_CONV_WARPS);
    if (!va) g.ka *= 2;
    g.bank_chunks = (long long)g.nu * t.ru * g.s * 2 * t.nt;
    return g;
}

int filter_tiles(const DirectProblem& pr, const F3Tile& t) { return t.r > 1 ? 1 : (pr.nf + t.nt - 1) / t.nt; }

long long virtual_width(const DirectProblem& pr) { return (long long)pr.out_w + pr.fw - 1; }

long long pixel_tiles(const DirectProblem& pr, const F3Tile& t) {
    return ((pr.out_h + t.r - 1) / t.r * virtual_width(pr) + 127) / 128;
}

// Ring depths: three to six A slots, and two B rings of the stages that then fit, up
// to 8 each (at least 3: a copy takes about 1 us).
bool layout(const DirectProblem& pr, const F3Tile& t, int* na, int* nb, size_t* smem) {
    if (t.ord < 1 || t.ord > 3 || t.nt < 16 || t.nt > (t.ord == 3 ? 80 : 96) || t.nt % 16 || t.r < 1 || t.ru < 1 || t.jt < 1 || t.jt > pr.fw)
        return false;
    if (t.gc != 8 && t.gc != 16 && t.gc != 32) return false;
    if (t.gc > 8 && pr.c <= 4) return false;
    if (t.r > 1 && (long long)t.r * pr.nf > t.nt) return false;
    if (t.ru > pr.fh + t.r - 1) return false;
    // 32-bit pixel indices, with room for a slab past the last tile
    if ((pixel_tiles(pr, t) + 1) * 128 + 4096 >= (1ll << 31)) return false;
    const Geometry g = geometry(pr, t);
    if (g.ka > 18 || g.bank_chunks >= (1ll << 30)) return false;
    for (int want : {4, 3})
        for (int a = 6; a >= 3; --a) {
            const long room = (long)kSmemMax - kBarBytes - (long)(a * g.aslot);
            const int b = room < 0 ? 0 : (int)std::min<long>(8, room / (long)(2 * g.bstage));
            if (b < want) continue;
            *na = a;
            *nb = b;
            *smem = a * g.aslot + 2 * b * g.bstage + kBarBytes;
            return true;
        }
    return false;
}

// Cycles of a launch, to rank tiles.  A K = 16 step takes 3 NT cycles of the tensor
// core, or longer at narrow tiles (measured alone: 123, 144, 168, 204, 244 cycles
// at NT = 16 .. 80); a unit measured 600 to 900 cycles more (barriers, commits, the
// drain that is not hidden).  The converters take for each pass
// over their threads about 170 cycles where a slab is a run of whole pixels, 290 where
// it takes some channels of deeper ones, 250 where a pixel's row has to be divided out
// (folded rows, dL/dx).  A finished tile's stores, 45 cycles a column (more where they
// are narrower than 32 bytes), are spread over a tile's units.
// shared: the launch runs beside others that fill the SMs its last round leaves idle.
double model_cycles(const DirectProblem& pr, const F3Tile& t, int sm_count, bool shared) {
    const Geometry g = geometry(pr, t);
    // (an MMA of N columns alone: the longer of N / 2 and 32 + N / 4 cycles)
    auto mma_cycles = [](int n) { return std::max(n / 2.0, 32 + n / 4.0); };
    const double step = t.ord == 3   ? std::max(102.0 + 1.2 * t.nt, 3.06 * t.nt)
                        : t.ord == 2 ? mma_cycles(2 * t.nt) + mma_cycles(t.nt)
                                     : mma_cycles(t.nt);
    const long long items = pixel_tiles(pr, t) * filter_tiles(pr, t);
    const double rounds = shared ? (double)items / sm_count : (double)((items + sm_count - 1) / sm_count);
    const double pass = t.r > 1 || pr.flip ? 250 : t.gc < pr.c ? 290 : 170;
    const double store = (pr.nf % 8 == 0 ? 45.0 : pr.nf % 4 == 0 ? 90.0 : 180.0) * t.nt / g.nu;
    const double mma = t.ru * g.s * step + 700, conv = pass * g.ka + 300, drain = 400.0 + 8 * t.nt + store;
    return rounds * g.nu * std::max(std::max(mma, conv), drain) + 4000;
}

// Steps summed on the tensor core before a chunk is added up in FP32.  Relative errors
// (2-norm, against 64 bits) measured with up to 16, this kernel / the FMA kernels, for
// random values: 128x128x8 * 16x9x9 1.9e-7 / 1.7e-7 (dL/dx 2.0e-7 / 6.3e-7),
// 256x256x8 * 64x9x9 1.9e-7 / 2.3e-7 (2.2e-7 / 1.3e-6), 2048x2048x4 * 4x8x8
// 1.4e-7 / 1.5e-7 (1.5e-7 / 2.8e-7), 512x512x32 * 256x5x5 1.4e-7 / 2.6e-7
// (2.2e-7 / 1.4e-6), 64x200x128 * 64x8x8 2.4e-7 / 1.6e-6 (2.4e-7 / 1.1e-6); on nine
// more shapes 3.5e-8 to 1.8e-7 / 6.5e-8 to 2.6e-7 (4.6e-8 to 2.1e-7 / 9.6e-8 to 1.3e-6).
constexpr int kChunkSteps = 16;

}  // namespace

std::string f3_spec(const F3Tile& t) {
    char b[96];
    snprintf(b, sizeof b, "%s:nt=%d,r=%d,gc=%d,jt=%d,ru=%d", t.ord == 3 ? "f32tc" : "tcpack", t.nt, t.r, t.gc, t.jt, t.ru);
    return b;
}

bool f3_parse_spec(const std::string& s, F3Tile* t, int ord) {
    F3Tile v;
    v.ord = ord;
    int used = 0;
    if (sscanf(s.c_str(), ord == 3 ? "f32tc:nt=%d,r=%d,gc=%d,jt=%d,ru=%d%n" : "tcpack:nt=%d,r=%d,gc=%d,jt=%d,ru=%d%n", &v.nt, &v.r, &v.gc, &v.jt, &v.ru, &used) != 5 ||
        used != (int)s.size())
        return false;
    *t = v;
    return true;
}

std::vector<F3Tile> f3_ranked(const DirectProblem& pr, int sm_count, double* best_cycles, bool shared, int ord) {
    const int chunk_steps = ord == 3 ? kChunkSteps : 2 * kChunkSteps;   // the BF16 modes never added up in between
    const int widest = ord == 3 ? 80 : 96;
    std::vector<std::pair<double, F3Tile>> all;
    const int npad = (pr.nf + 15) / 16 * 16;
    for (int fold = 1; fold <= std::min(16, pr.out_h); ++fold) {
        if (fold > 1 && fold * pr.nf > widest) break;
        F3Tile t;
        t.ord = ord;
        t.r = fold;
        const int ntn = (npad + widest - 1) / widest;
        t.nt = fold > 1 ? (fold * pr.nf + 15) / 16 * 16 : ((npad + ntn - 1) / ntn + 15) / 16 * 16;
        for (int gc : {32, 16, 8}) {   // no whole group of padding
            if (gc > 8 && (pr.c <= 4 || pr.c <= gc / 2)) continue;
            t.gc = gc;
            for (int ntg = 1, jt = 0; ntg <= pr.fw; ++ntg) {
                t.jt = (pr.fw + ntg - 1) / ntg;
                if (t.jt == jt) continue;
                jt = t.jt;
                t.ru = 1;
                const Geometry g = geometry(pr, t);
                if (g.s > chunk_steps) continue;
                // slab rows per unit, evenly, within the chunk length and half of it
                for (int steps : {chunk_steps, chunk_steps / 2}) {
                    const int most = std::max(1, std::min(g.rows, steps / g.s)), units = (g.rows + most - 1) / most;
                    const int ru = (g.rows + units - 1) / units;
                    if (steps != chunk_steps && ru == t.ru) break;
                    t.ru = ru;
                    int na, nb;
                    size_t smem;
                    if (!layout(pr, t, &na, &nb, &smem)) continue;
                    // three A slots measured 5 % behind four or more
                    all.push_back({model_cycles(pr, t, sm_count, shared) * (na < 4 ? 1.06 : 1.0), t});
                }
                if (g.s <= 4) break;   // splitting the taps further only adds slabs
            }
        }
    }
    std::stable_sort(all.begin(), all.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
    std::vector<F3Tile> out;
    for (const auto& a : all) out.push_back(a.second);
    if (best_cycles) *best_cycles = all.empty() ? 0 : all.front().first;
    return out;
}

// The line between the two FP32 kernels: the model's cycles and the bank split's
// launch (about 9000 cycles, 5 us) against the FMA kernels at 0.55 of their peak (the
// forward; 0.65 at size, in a batch) or 0.35 (dL/dx of the untuned tiles).  Measured
// (us, FMA kernel / this one): 128x128x8 * 16x9x9 (0.3 GFLOP) 11 / 19, 187x233x12 *
// 40x5x3 (0.6) 20 / 20, 256x256x8 * 64x9x9 (5.1) 115 / 34, 2048x2048x4 * 4x8x8 (8.5)
// 180 / 92, 512x512x32 * 256x5x5 (106) 1935 / 428.
// Beside other launches (shared) neither the launch nor the last round counts.
bool f3_wins(const DirectProblem& pr, int sm_count, F3Tile* t, bool shared) {
    const std::string sw = env_str("FBCORR_F32TC", "1");
    if (sw == "0") return false;
    double cycles = 0;
    const std::vector<F3Tile> r = f3_ranked(pr, sm_count, &cycles, shared);
    if (r.empty()) return false;
    *t = r.front();
    const double flops = 2.0 * pr.out_h * pr.out_w * pr.nf * pr.fh * pr.fw * pr.c;
    const double eff = shared ? 0.65 : pr.flip ? 0.35 : 0.55;
    return sw == "force" || cycles + (shared ? 0 : 9000) < 0.9 * (flops / (sm_count * 256 * eff) + (shared ? 0 : 4000));
}

// The BF16 modes' own kernel (rtcg_tc.cuh) measured 1.35 of its MMAs' time and about
// 1400 cycles per filter row and 128-pixel tile: far from the tensor rate where the
// rows are short (narrow banks, shallow or ragged depths, which it pads to 16).
// Measured untuned (GB300, us, that kernel / this one, split BF16): 244x244x32 *
// 16x3x3 21 / 10, 400x400x16 * 128x3x3 33 / 37, 256x256x8 * 64x9x9 60 / 26, 248x248x64 * 32x5x5 62 / 33, 300x500x32
// * 64x7x7 124 / 77, 512x512x4 * 32x13x13 361 / 38, 2048x2048x4 * 4x8x8 2287 / 74;
// 200x300x32 * 128x5x5 40 / 44.
bool f3_wins_bf16(const DirectProblem& pr, int sm_count, int ord, size_t ws_limit, F3Tile* t) {
    if (env_str("FBCORR_TCPACK", "1") == "0" || fault_injected("tcdrop")) return false;
    double cycles = 0;
    const std::vector<F3Tile> r = f3_ranked(pr, sm_count, &cycles, false, ord);
    if (r.empty() || f3_ws_bytes(pr, r.front()) > ws_limit) return false;
    *t = r.front();
    const int npad = (pr.nf + 15) / 16 * 16, ntn = (npad + 255) / 256, nt = ((npad + ntn - 1) / ntn + 15) / 16 * 16;
    const double tiles = ((double)pr.out_h * pr.in_w / 128 + 1) * ntn;
    const double rounds = std::max(1.0, tiles > 4 * sm_count ? tiles / sm_count : std::ceil(tiles / sm_count));
    const double mma = (double)pr.fw * ((pr.c + 15) / 16) * (ord == 2 ? 3 : 1) * std::max(nt / 2.0, 32 + nt / 4.0);
    const double tc = rounds * pr.fh * (1.35 * mma + 1400) + 4000;
    // the margin keeps near ties on their own kernel: BF16 301x419x24 * 96x7x5 47 / 53
    return cycles + 2000 < 0.75 * tc;
}

size_t f3_ws_bytes(const DirectProblem& pr, const F3Tile& t) {
    int na, nb;
    size_t smem;
    if (!layout(pr, t, &na, &nb, &smem)) return 0;
    const Geometry g = geometry(pr, t);
    return (size_t)filter_tiles(pr, t) * g.nu * g.bunit;
}

std::string f3_kernel_name(const DirectProblem& pr, const F3Tile& t) {
    char b[160];
    snprintf(b, sizeof b, "%s_f%dx%d_c%d_n%d_fl%d_e%d_m%d_t%d_%d_%d_%d_%d", t.ord == 3 ? "fbc_f32tc" : t.ord == 2 ? "fbc_tcpack2" : "fbc_tcpack1", pr.fh, pr.fw, pr.c, pr.nf, pr.flip,
             pr.epi, pr.mask, t.nt, t.r, t.gc, t.jt, t.ru);
    const std::string name = b;
    return pr.epi == 2 ? name + "_u" + snippet_tag(pr.snippet) : name;
}

std::string f3_kernel_source(const DirectProblem& pr, const F3Tile& t, const std::string& name) {
    std::ostringstream o;
    if (fault_injected("f3drop")) o << "#define FBC_F3_DROP 1\n";   // tests: the first bank copy never comes
    o << rtcg_f32tc_params_source() << "\n" << rtcg_ptx_source() << "\n" << rtcg_f32tc_source() << "\n"
      << snippet_definition(pr.epi == 2 ? pr.snippet : "");
    o << "static_assert(sizeof(FbcF3Params) == " << sizeof(FbcF3Params)
      << ", \"host and device disagree on the parameter block\");\n";
    const Geometry g = geometry(pr, t);
    o << "typedef FbcF3Cfg<" << pr.fh << "," << pr.fw << "," << pr.c << "," << pr.nf << "," << pr.flip << "," << pr.epi
      << "," << pr.mask << "," << t.nt << "," << t.r << "," << t.gc << "," << t.jt << "," << t.ru
      << "," << t.ord << "> FbcF3;\nstatic_assert(FbcF3::ASLOT == " << g.aslot << " && FbcF3::BSTAGE == " << g.bstage
      << " && FbcF3::NU == " << g.nu << ", \"host and device disagree on the geometry\");\n";
    o << "extern \"C\" __global__ void __launch_bounds__(" << FBC_F3_THREADS << ", 1) " << name
      << "(const __grid_constant__ FbcF3Params P) {\n"
      << "  fbc_f32tc_body<FbcF3>(P);\n}\n";
    o << "extern \"C\" __global__ void __launch_bounds__(" << FBC_F3_BANK_THREADS << ") " << name
      << "_bank(const __grid_constant__ FbcF3Params P) {\n  fbc_f32tc_bank_body<FbcF3>(P);\n}\n";
    return o.str();
}

fbcorr_status_t f3_build(const DirectProblem& pr, const F3Tile& t, int sm_count, F3Launch* out) {
    F3Launch l;
    size_t smem = 0;
    if (!layout(pr, t, &l.na, &l.nb, &smem))
        return set_error(FBCORR_ERR_UNSUPPORTED, "variant %s does not fit this shape", f3_spec(t).c_str());
    l.tile = t;
    const Geometry g = geometry(pr, t);
    const std::string name = f3_kernel_name(pr, t), src = f3_kernel_source(pr, t, name);
    FBC_TRY(rtcg_kernel(src, name, smem, FBC_F3_THREADS, &l.kernel));
    FBC_TRY(rtcg_second_kernel(l.kernel, name + "_bank", 0, FBC_F3_BANK_THREADS, &l.bank));
    l.filter_tiles = filter_tiles(pr, t);
    const long long items = pixel_tiles(pr, t) * l.filter_tiles;
    l.grid = (int)std::min<long long>(items, std::max(1, sm_count));
    l.bank_blocks = (int)((g.bank_chunks + FBC_F3_BANK_THREADS - 1) / FBC_F3_BANK_THREADS);
    l.ws_bytes = f3_ws_bytes(pr, t);
    l.wait_ns = wait_bound_ns();
    *out = l;
    return FBCORR_OK;
}

FbcF3Params f3_params(const F3Launch& l, const DirectProblem& pr, const float* x, const float* m, const float* w,
                      float* y, void* ws, float lo, float hi, int* err_word) {
    const Geometry g = geometry(pr, l.tile);
    FbcF3Params k;
    memset(&k, 0, sizeof k);
    k.x = x; k.m = m; k.w = w; k.y = y;
    k.bank = static_cast<unsigned char*>(ws);
    k.err = err_word;
    k.wait_ns = l.wait_ns;
    k.lo = lo; k.hi = hi;
    k.in_h = pr.in_h; k.in_w = pr.in_w; k.out_h = pr.out_h; k.out_w = pr.out_w;
    k.pad_y = pr.pad_y; k.pad_x = pr.pad_x;
    k.vw = (int)virtual_width(pr);
    // division of 31-bit numbers by vw > 1 (Granlund and Montgomery, "Division by
    // invariant integers using multiplication"): with 2^(l-1) < vw <= 2^l,
    // floor(2^(31+l) / vw) + 1 fits in 32 bits
    int lg = 0;
    while ((1ll << lg) < k.vw) ++lg;
    k.vw_mul = k.vw > 1 ? (unsigned)((1ull << (31 + lg)) / (unsigned)k.vw + 1) : 0u;
    k.vw_shift = lg - 1;
    k.mtiles = (int)pixel_tiles(pr, l.tile);
    k.nitems = k.mtiles * l.filter_tiles;
    k.na = l.na; k.nb = l.nb;
    k.b_off = (unsigned)(l.na * g.aslot);
    k.bar_off = (unsigned)(k.b_off + 2 * l.nb * g.bstage);
    return k;
}

dim3 f3_bank_grid(const F3Launch& l) { return dim3((unsigned)l.bank_blocks, (unsigned)l.filter_tiles); }

fbcorr_status_t f3_run(const F3Launch& l, const DirectProblem& pr, const float* x, const float* m, const float* w,
                       float* y, void* ws, float lo, float hi, int* err_word, cudaStream_t s) {
    FbcF3Params k = f3_params(l, pr, x, m, w, y, ws, lo, hi, err_word);
    void* args[] = {&k};
    FBC_TRY(launch_dependent(l.bank, f3_bank_grid(l), args, s));
    return launch_dependent(l.kernel, dim3(l.grid), args, s);
}

std::vector<F3Tile> f3_candidates(const DirectProblem& pr, int sm_count, int ord, size_t ws_limit) {
    if (env_str(ord == 3 ? "FBCORR_F32TC" : "FBCORR_TCPACK", "1") == "0") return {};
    std::vector<F3Tile> tiles = f3_ranked(pr, sm_count, nullptr, false, ord);
    tiles.erase(std::remove_if(tiles.begin(), tiles.end(), [&](const F3Tile& t) { return f3_ws_bytes(pr, t) > ws_limit; }),
                tiles.end());
    tiles.resize(std::min<size_t>(tiles.size(), 8));
    return tiles;
}

fbcorr_status_t f3_tune(const DeviceInfo& dev, const DirectProblem& pr, cudaStream_t s, int* err_word, float* ms,
                        std::string* spec, int ord, size_t ws_limit) {
    spec->clear();
    const std::vector<F3Tile> tiles = f3_candidates(pr, dev.sm_count, ord, ws_limit);
    if (tiles.empty()) return FBCORR_OK;
    std::vector<std::string> srcs;
    for (const F3Tile& t : tiles) srcs.push_back(f3_kernel_source(pr, t, f3_kernel_name(pr, t)));
    rtcg_precompile(srcs);
    const size_t xn = (size_t)pr.in_h * pr.in_w * pr.c, wn = (size_t)pr.nf * pr.fh * pr.fw * pr.c,
                 yn = (size_t)pr.out_h * pr.out_w * pr.nf;
    size_t wsn = 0;
    for (const F3Tile& t : tiles) wsn = std::max(wsn, f3_ws_bytes(pr, t));
    float *x = nullptr, *w = nullptr, *y = nullptr, *m = nullptr;
    void* ws = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    fbcorr_status_t status = FBCORR_OK;
    if (cudaMalloc(&x, xn * 4) != cudaSuccess || cudaMalloc(&w, wn * 4) != cudaSuccess ||
        cudaMalloc(&y, yn * 4) != cudaSuccess || scratch_alloc(&ws, wsn) != cudaSuccess ||
        (pr.mask && cudaMalloc(&m, xn * 4) != cudaSuccess) || cudaEventCreate(&e0) != cudaSuccess ||
        cudaEventCreate(&e1) != cudaSuccess) {
        cudaGetLastError();
        logf("no memory to time the tensor-core tiles: the other variants are left");
    } else {
        launch_fill_pattern(x, xn, 1.0f, 0x1234u, s);
        launch_fill_pattern(w, wn, 0.05f, 0x5678u, s);
        if (m) launch_fill_pattern(m, xn, 1.0f, 0x9abcu, s);
        // best of three rounds of ten back-to-back calls, round-robin
        std::vector<float> best(tiles.size(), 1e30f);
        for (int round = 0; round < 3 && status == FBCORR_OK; ++round)
            for (size_t k = 0; k < tiles.size(); ++k) {
                F3Launch l;
                if (f3_build(pr, tiles[k], dev.sm_count, &l) != FBCORR_OK) continue;
                bool ok = true;
                for (int r = 0; r < 12 && ok; ++r) {
                    if (r == 2) cudaEventRecord(e0, s);
                    ok = f3_run(l, pr, x, m, w, y, ws, 0.f, 1.f, err_word, s) == FBCORR_OK;
                }
                cudaEventRecord(e1, s);
                float t = 0.f;
                if (!ok || cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) {
                    status = set_error(FBCORR_ERR_CUDA, "autotune run of %s failed", f3_spec(tiles[k]).c_str());
                    break;
                }
                best[k] = std::min(best[k], t / 10.f);
            }
        for (size_t k = 0; k < tiles.size() && status == FBCORR_OK; ++k) {
            logf("autotune %s: %.4f ms", f3_spec(tiles[k]).c_str(), best[k]);
            if (best[k] < 1e30f && (spec->empty() || best[k] < *ms)) {
                *ms = best[k];
                *spec = f3_spec(tiles[k]);
            }
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(x); cudaFree(w); cudaFree(y); cudaFree(m); cudaFree(ws);
    return status;
}

}  // namespace fbc

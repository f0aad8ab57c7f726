// f32dw_kernel.cu -- host side of the FP32 tensor-core dL/dw kernel
// (rtcg_f32dw.cuh): tile and split selection, run-time generation, launch.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <sstream>

#include "f32dw_params.h"
#include "internal.h"

namespace fbc {

namespace {

// The kernel template's derived constants (FbcF3DwCfg of rtcg_f32dw.cuh).
struct DwGeometry {
    int fwp, nn, ntg, ncp, ntn, nh, steps, mmas;
    size_t slot;
    int ns;
};

DwGeometry geometry(const DirectProblem& pr, const F3DwTile& t) {
    DwGeometry g;
    g.fwp = (t.jt + 1) / 2 * 2;
    g.nn = 8 * g.fwp;
    g.ntg = (pr.fw + t.jt - 1) / t.jt;
    g.ncp = (pr.c + 8 * t.ncomb - 1) / (8 * t.ncomb);
    g.ntn = (pr.nf + t.nb - 1) / t.nb;
    g.nh = t.nb == 64 ? 2 : 3;
    g.steps = t.kpx / 16;
    g.mmas = t.nb == 64 ? 4 : 3;
    const size_t gplane = (size_t)t.kpx * 16 + 16, gplanes = t.nb == 64 ? 32 : 16;
    const int ls = t.kpx + g.fwp - 1, lp = t.ncomb == 2 ? (ls + 3) / 8 * 8 + 4 : ls;
    g.slot = (gplanes * gplane + (size_t)3 * t.ncomb * lp * 16 + 127) / 128 * 128;
    const size_t room = 227 * 1024 - 2048;
    g.ns = room >= 4 * g.slot ? 4 : room >= 3 * g.slot ? 3 : 2;
    return g;
}

long chunks(const DirectProblem& pr, const F3DwTile& t) {
    return ((long)pr.out_h * pr.in_w + t.kpx - 1) / t.kpx;
}

long combos(const DirectProblem& pr, const F3DwTile& t) {
    const DwGeometry g = geometry(pr, t);
    return (long)pr.fh * g.ntg * g.ncp * g.ntn;
}

// Cycles of a chunk: the MMAs (36 to 64 cycles at N = 16 .. 128, measured alone) or
// the drain of the accumulators, and of a CTA's start and end.
double chunk_cycles(const DirectProblem& pr, const F3DwTile& t) {
    const DwGeometry g = geometry(pr, t);
    return std::max(1.15 * g.steps * t.ncomb * g.mmas * (32.0 + g.nn / 4.0), 700.0 + 3.0 * t.ncomb * g.nn) + 150;
}
constexpr double kCtaCycles = 5000;

}  // namespace

size_t f3dw_ws_bytes(const DirectProblem& pr, const F3DwTile& t) {
    const size_t part = (size_t)t.splits * geometry(pr, t).nh * pr.nf * pr.fh * pr.fw * pr.c * 4;
    return (part + 255) / 256 * 256 + (size_t)combos(pr, t) * t.splits * sizeof(int);
}

// Whether the tensor cores are expected to be faster than the FMA kernel (0.45 of
// its peak), and the tile: 64 filters per tile, 32 where the bank is no
// wider; two planes of x per CTA where their accumulators fit in TMEM twice; as
// many CTAs as fill whole rounds of the SMs.  Needs 16-byte rows of x and g.
// Measured (GB300, us, FMA / this): 187x233x12 * 40x5x3 34 / 28 (not taken; clamped 40 /
// 31), 256x256x8 * 64x9x9 113 / 56 (137 / 70), 256x256x16 * 64x7x7 125 / 60 (151 / 60),
// 40x300x64 * 100x3x11 112 / 59 (132 / 75), 512x512x32 * 256x5x5 2141 / 1034 (2597 / 1098),
// 2048x2048x4 * 4x8x8 3223 / 1796 (7243 / 2016).  Of 130 drawn shapes it takes 82, four of
// them wrongly, all with at most 16 filters, which fill half of a tile of 32 or less:
// 756x191x16 * 8x2x7 36.9 / 37.4, 463x114x64 * 16x9x9 clamped 214 / 230, 666x254x16 *
// 4x9x9 154 / 184, 254x72x16 * 16x11x11 27.5 / 35.6; lines that leave these out lose as
// much on others (973x135x12 * 16x3x3 46 / 38, 51x1065x12 * 4x3x8 clamped 73 / 26).
bool f3dw_wins(const DirectProblem& pr, int sm_count, F3DwTile* out) {
    const std::string sw = env_str("FBCORR_F32TC", "1");
    if (sw == "0" || pr.c % 4 || pr.nf % 4 || pr.c > 256) return false;
    if ((long)pr.in_h * pr.in_w + pr.fw + 512 >= (1l << 31) / std::max(1, pr.c)) return false;
    F3DwTile t;
    t.nb = pr.nf <= 32 ? 32 : 64;
    t.kpx = t.nb == 64 ? 96 : 128;
    const int ntg = (pr.fw + 15) / 16;
    t.jt = (pr.fw + ntg - 1) / ntg;
    t.ncomb = pr.c > 8 && (t.jt + 1) / 2 * 2 <= 8 ? 2 : 1;
    const DwGeometry g = geometry(pr, t);
    const long nchunk = chunks(pr, t), nc = combos(pr, t);
    const size_t elems = (size_t)pr.nf * pr.fh * pr.fw * pr.c;
    double best = -1;
    // at most 256 partial sums per element (what the reduction takes) and 64 MB of them
    for (long s = 1; s <= std::min<long>(256 / g.nh, nchunk) && (size_t)s * g.nh * elems * 4 <= (64u << 20); ++s) {
        const double rounds = (double)((nc * s + sm_count - 1) / sm_count);
        const double cyc = rounds * ((double)((nchunk + s - 1) / s) * chunk_cycles(pr, t) + kCtaCycles) +
                           (double)s * g.nh * elems * 8 / 2000;
        if (best < 0 || cyc < best) {
            best = cyc;
            t.splits = (int)s;
        }
    }
    if (best < 0) return false;
    *out = t;
    const double flops = 2.0 * pr.out_h * pr.out_w * pr.nf * pr.fh * pr.fw * pr.c;
    // the FMA kernel's CTA has a thread per channel and 4 or 8 filters: a few threads
    // where both are few (2048x2048x4 * 4x8x8: four, 0.04 of the peak)
    const int tn = pr.c <= 64 && !pr.mask ? 8 : 4;
    const int threads = pr.c * std::max(1, std::min((tn == 8 ? 128 : 256) / pr.c, (pr.nf + tn - 1) / tn));
    const double eff = 0.45 * std::min(1.0, threads / 64.0);
    return sw == "force" || best + 5000 < 0.9 * (flops / (sm_count * 256 * eff) + 4000);
}

std::string f3dw_kernel_source(const DirectProblem& pr, const F3DwTile& t, std::string* kname) {
    const DwGeometry g = geometry(pr, t);
    char name[160];
    snprintf(name, sizeof name, "fbc_f32dw_f%dx%d_c%d_n%d_m%d_t%d_%d_%d_%d", pr.fh, pr.fw, pr.c, pr.nf, pr.mask, t.nb, t.ncomb,
             t.jt, t.kpx);
    std::ostringstream o;
    if (fault_injected("f3drop")) o << "#define FBC_F3_DROP 1\n";   // tests: the first chunk is never handed over
    o << rtcg_f32tc_params_source() << "\n" << rtcg_f32dw_params_source() << "\n" << rtcg_ptx_source() << "\n"
      << rtcg_f32tc_source() << "\n" << rtcg_f32dw_source() << "\n";
    o << "static_assert(sizeof(FbcF3DwParams) == " << sizeof(FbcF3DwParams)
      << ", \"host and device disagree on the parameter block\");\n";
    o << "typedef FbcF3DwCfg<" << pr.fh << "," << pr.fw << "," << pr.c << "," << pr.nf << "," << pr.mask << "," << t.nb << ","
      << t.ncomb << "," << t.jt << "," << t.kpx << "> FbcF3Dw;\nstatic_assert(FbcF3Dw::SLOT == " << g.slot
      << " && FbcF3Dw::NS == " << g.ns << " && 2 * FbcF3Dw::BUF <= 512, \"host and device disagree on the geometry\");\n";
    o << "extern \"C\" __global__ void __launch_bounds__(" << FBC_F3DW_THREADS << ", 1) " << name
      << "(const __grid_constant__ FbcF3DwParams P) {\n  fbc_f32dw_body<FbcF3Dw>(P);\n}\n";
    *kname = name;
    return o.str();
}

fbcorr_status_t f3dw_build(const DirectProblem& pr, const F3DwTile& t, F3DwLaunch* out) {
    const DwGeometry g = geometry(pr, t);
    std::string name;
    const std::string src = f3dw_kernel_source(pr, t, &name);
    F3DwLaunch l;
    l.tile = t;
    FBC_TRY(rtcg_kernel(src, name, g.ns * g.slot, FBC_F3DW_THREADS, &l.kernel));
    l.grid = (int)(combos(pr, t) * t.splits);
    l.parts = t.splits * g.nh;
    l.ws_bytes = f3dw_ws_bytes(pr, t);
    l.wait_ns = wait_bound_ns();
    *out = l;
    return FBCORR_OK;
}

fbcorr_status_t f3dw_run(const F3DwLaunch& l, const DirectProblem& pr, const float* x, const float* g, const float* m,
                         void* ws, float lo, float hi, int* err_word, const float** part, const int** flags,
                         cudaStream_t s) {
    FbcF3DwParams k;
    memset(&k, 0, sizeof k);
    k.x = x; k.g = g; k.m = m;
    k.part = static_cast<float*>(ws);
    const size_t part_bytes = (size_t)l.parts * pr.nf * pr.fh * pr.fw * pr.c * 4;
    k.flags = reinterpret_cast<int*>(static_cast<uint8_t*>(ws) + (part_bytes + 255) / 256 * 256);
    k.err = err_word;
    k.wait_ns = l.wait_ns;
    k.lo = lo; k.hi = hi;
    k.H = pr.in_h; k.W = pr.in_w; k.Ho = pr.out_h; k.Wo = pr.out_w;
    int lg = 0;
    while ((1ll << lg) < k.W) ++lg;      // as in f3_params
    k.w_mul = k.W > 1 ? (unsigned)((1ull << (31 + lg)) / (unsigned)k.W + 1) : 0u;
    k.w_shift = lg - 1;
    k.nchunk = (int)chunks(pr, l.tile);
    k.splits = l.tile.splits;
    *part = k.part;
    *flags = k.flags;
    void* args[] = {&k};
    return launch(l.kernel, dim3((unsigned)l.grid), args, s);
}

}  // namespace fbc

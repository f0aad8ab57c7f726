// rtcg_f32tc.cuh -- the FP32 correlation on the tensor cores, compiled at plan
// time by NVRTC for sm_103a.  Embedded as a string into libfbcorr and prefixed
// with f32tc_params.h and rtcg_ptx.cuh; self-contained (no system headers).
//
// Arithmetic.  Every FP32 operand is split exactly into three BF16 values,
// v = v1 + v2 + v3 with v1 = bf16_rn(v), v2 = bf16_rn(v - v1), v3 = v - v1 - v2
// (24 significand bits in three 8-bit ones), and the product x w is taken as the
// six largest of the nine BF16 products, each exact in FP32:
//   order 0: x1 w1      order 1: x1 w2 + x2 w1      order 2: x1 w3 + x2 w2 + x3 w1
// The three that are left out are together below 2^-24 |x w| (|v2| <= 2^-8 |v| and
// |v3| <= 2^-17 |v|: x2 w3 and x3 w2 up to 2^-25 each).  The tensor core truncates
// its FP32 accumulator at every K = 16 step, so a sum is only left there for a
// chunk of a few steps: each order has its own accumulator (a truncation of
// order 1 and 2 is then 2^-8 and 2^-16 below one of the result), and the chunk
// sums are added to FP32 registers with ordinary rounding.  Measured errors against
// 64 bits, beside the FMA kernels' on the same values: kChunkSteps in f32tc_kernel.cu.
//
// ORD is the number of orders: 3 for FP32.  The BF16 modes run the same kernel with
// fewer where their own one (rtcg_tc.cuh) is far from the tensor rate: ORD = 2 is
// split BF16 (x1 w1, x1 w2 + x2 w1), ORD = 1 plain BF16.
//
// Layout.  As in the BF16 kernels, an A tile is 128 consecutive pixels of the
// image laid out with the virtual row width vw = out_w + FW - 1 (columns past
// out_w are computed and dropped), and one slab of pixels serves every filter
// tap of a row: tap j is the slab started j pixels later.  The three orders of B
// lie side by side as 3 NT rows of one operand, so a K = 16 step is three MMAs,
//   x1 x [w1 w2 w3] (N = 3 NT) -> columns [0, 3 NT)
//   x2 x [w1 w2]    (N = 2 NT) -> columns [NT, 3 NT)
//   x3 x [w1]       (N =   NT) -> columns [2 NT, 3 NT)
// which read each A tile three times instead of six: at NT = 64 the operand
// reads of shared memory (24 KB per step) take as long as the MMAs (192 cycles).
//
// Depth.  GC = 16 or 32: the step takes 16 channels of one tap (two chunk
// planes of 8 channels, LBO = one plane).  GC = 8: one plane whose 16-byte chunk
// at pixel q holds PP = 8 / CP pixels q .. q + PP - 1 of CP channels, and the
// second half of the step is the same plane PP pixels later (LBO = 16 PP bytes):
// a step covers 2 PP taps, so depths of 1, 2, 4 and 8 waste none of K = 16.
//
// Rows.  R > 1 (narrow banks): the columns of B are R output rows x NF filters,
// column (r, n) of slab row u holding filter row u - r (zero outside the
// filter), so one slab row feeds R output rows and FH + R - 1 rows of MMAs do the
// work of R FH.
//
// Units.  A unit is RU slab rows of one channel and tap group; its RU S steps are
// one accumulation chunk, its A slot holds RU slabs and its B stage all filters of
// the tile.  The bank is split once per call (fbc_f32tc_bank_body) into the images
// of the B stages, so that a stage is one bulk copy.
//
// Roles per CTA (persistent, one per SM): warps 0..7 add the chunk sums up and
// store; warps 8..12 read x from global memory (prefetched in registers), split it
// and write the A slots; a thread of warp 13 copies the B stages; a thread of
// warp 14 issues the MMAs of every other unit, one of warp 15 the rest, each from
// its own B ring into its own accumulator set, so chunk sums are drained while the
// next chunk runs.  (A barrier is only ever waited for by threads that have seen its
// phase before: the parity does not tell phase k from k - 2.  B stages therefore
// have one ring per issuer; A slots, which the converters fill in order, do not need
// it: an issuer that has seen unit u - 2 filled knows that every earlier one was.)
//
// Range.  BF16 has the exponents of FP32, so the third part of a |v| below 2^-110
// would fall out of its range, and so would products near 2^-126.  FP32 operands are
// therefore split as 2^16 v (the least bit of any FP32 value, 2^-149, becomes the
// least one of BF16, 2^-133) and the sums multiplied by 2^-32 at the end, both exact
// but for results below the normal range: every value splits exactly, and the small
// orders keep their bits where FP32 keeps those of the result.  Before, one such value
// sent its tiles (one in the bank: all of them) to the FMAs below: 512x512x32 *
// 256x5x5 with one tiny weight took 79 ms, now 0.4 as without it (0.7 % more than with
// the unscaled split; 2048x2048x4 * 4x8x8 9 % less, as nothing is searched for).
//
// Values the split cannot carry.  Non-finite inputs, and sums from 2^96, give a
// non-finite sum.  The epilogue warps only note where (a call in their loop cost
// 2048x2048x4 * 4x8x8 a fifth in spilled registers); once the pipeline has ended, all
// warps of the CTA compute those outputs again, in groups of 8 pixels x 8 columns, with
// FP32 FMAs straight from global memory (fbc_f3_redo_noted).
//
// Every mbarrier wait is bounded in time; on expiry the kernel records an error
// code in host-mapped memory, stops every role, waits (bounded) for its MMAs in
// flight, frees TMEM and returns.

#define FBC_F3_ERR_WAIT 5

// 1 (tests of the bounded waits): an arrival that the MMA issuers wait for never comes.
#ifndef FBC_F3_DROP
#define FBC_F3_DROP 0
#endif

// The PTX that the FP32 kernels alone use (the rest: rtcg_ptx.cuh, which is part of
// every kernel's source and of the hash that measured traffic is filed under).
// mbarrier test of a phase without a wait.
__device__ __forceinline__ bool fbc_mbar_test(fbc_u32 bar, fbc_u32 parity) {
    fbc_u32 ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// tcgen05.ld 32x32b.x8 -- 32 TMEM lanes x 8 columns, one accumulator row per thread.
__device__ __forceinline__ void fbc_tmem_ld32x32b_x8_async(fbc_u32 taddr, fbc_u32 (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void fbc_reg_fence8(fbc_u32 (&r)[8]) {
    asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
}

// 8-byte shared store.
__device__ __forceinline__ void fbc_st_shared_v2(fbc_u32 addr, fbc_u32 a, fbc_u32 b) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

// tcgen05.mma with the descriptors as low and high words.
__device__ __forceinline__ void fbc_umma_lo(fbc_u32 d, fbc_u32 alo, fbc_u32 ahi, fbc_u32 blo, fbc_u32 bhi, fbc_u32 idesc,
                                            fbc_u32 accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(d),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(accumulate));
}

// Snippet epilogue (EPI = 2): defined by the generated source after this file.
__device__ float fbc_user_epi(float y, int n, float lo, float hi);

template <int FH_, int FW_, int C_, int NF_, int FLIP_, int EPI_, int MASK_, int NT_, int R_, int GC_,
          int JT_, int RU_, int ORD_ = 3>
struct FbcF3Cfg {
    static constexpr int FH = FH_, FW = FW_, C = C_, NF = NF_, FLIP = FLIP_, EPI = EPI_, MASK = MASK_;
    static constexpr int NT = NT_, R = R_, GC = GC_, JT = JT_, RU = RU_, ORD = ORD_;
    static constexpr bool PACK = GC == 8;
    static constexpr int PP = !PACK ? 1 : C <= 1 ? 8 : C <= 2 ? 4 : C <= 4 ? 2 : 1;   // pixels per chunk
    static constexpr int CP = 8 / PP;                                                // channels per pixel in it
    static constexpr int PL = PACK ? 1 : GC / 8;                                     // chunk planes of a slab
    static constexpr int S = PACK ? (JT + 2 * PP - 1) / (2 * PP) : JT * (GC / 16);   // K = 16 steps per slab
    static constexpr int NCG = (C + GC - 1) / GC;                                    // channel groups
    static constexpr int NTG = (FW + JT - 1) / JT;                                   // tap groups
    static constexpr int ROWS = FH + R - 1;                                          // slab rows per pixel tile
    static constexpr int NU = (ROWS + RU - 1) / RU * NCG * NTG;                      // units per pixel tile
    static constexpr int LS = PACK ? 128 + (2 * S - 1) * PP : 128 + JT - 1;          // slab pixels
    // plane pitch in pixels: planes 32 (four planes) or 64 (two) bytes apart modulo
    // 128, so that the writes of neighbouring quads of a pixel hit other banks
    static constexpr int LP = PL == 4 ? (LS + 5) / 8 * 8 + 2 : PL == 2 ? (LS + 3) / 8 * 8 + 4 : LS;
    static constexpr unsigned PLANE = LP * 16;
    static constexpr unsigned AORD = PL * PLANE;                                     // bytes of one order of a slab
    static constexpr unsigned SLAB = ORD * AORD;
    static constexpr unsigned ASLOT = (RU * SLAB + 127) / 128 * 128;
    static constexpr unsigned BCH = ORD * NT * 16;             // bytes per chunk of B
    static constexpr unsigned BSTEP = 2 * BCH;
    static constexpr int STEPS = RU * S;                     // steps of a unit
    // a B stage holds BS steps, about 12 KB (one copy at the copy unit's full rate):
    // refills start, and are waited for, in small pieces
    static constexpr int BS = ORD * NT >= 144 ? 2 : ORD * NT >= 96 ? 4 : 8;
    static constexpr int NST = (STEPS + BS - 1) / BS;        // stages of a unit
    static constexpr unsigned BSTAGE = BS * BSTEP;
    static constexpr unsigned BUNIT = STEPS * BSTEP;         // the unit's image in the split bank
    static constexpr int NCT = 32 * FBC_F3_CONV_WARPS;
    // Items of the converters: quads of 4 channels read with one 16-byte load, lanes
    // along the channels, or (depths that are no multiple of 4) chunks of 8 single
    // loads, lanes along the pixels.
    static constexpr bool VA = C % 4 == 0;
    static constexpr int WA = VA ? 4 : 8;                    // floats per item
    static constexpr int QA = !VA ? PL : PP == 2 ? 1 : GC / 4;      // items per pixel
    static constexpr int NPX = VA && PP == 2 ? LS + 1 : LS;         // pixels read per slab
    static constexpr int NIT = RU * NPX * QA;                // items per unit
    static constexpr int KA = (NIT + NCT - 1) / NCT;
    // Clamp masks stay beside their values until these are written (where both fit):
    // compared as they were loaded, each load was waited for in turn (dL/dx of
    // 2048x2048x4 * 4x8x8, clamped: 228 to 104 us; FMA kernel 182).
    static constexpr bool LATE = MASK && 2 * KA * WA <= 72;
    static constexpr int RA = KA * WA * (LATE ? 2 : 1);      // registers of a unit
    static constexpr int PA = RA <= 18 ? 4 : RA <= 24 ? 3 : RA <= 36 ? 2 : 1;   // units in registers
    static constexpr int NBC = RU * S * 2 * NT;              // bank chunks per unit
    __device__ static __forceinline__ int tap_group(int u) { return NTG > 1 ? u % NTG : 0; }
    __device__ static __forceinline__ int channel_group(int u) { return NCG > 1 ? (u / NTG) % NCG : 0; }
    __device__ static __forceinline__ int row0(int u) { return u / (NTG * NCG) * RU; }
    static constexpr int TC = 2 * ORD * NT;                  // columns of the two accumulator sets
    static constexpr unsigned TMEM = TC <= 32 ? 32 : TC <= 64 ? 64 : TC <= 128 ? 128 : TC <= 256 ? 256 : 512;
};

#define FBC_F3_UP 65536.f                      // 2^16, of each operand of the FP32 split
#define FBC_F3_DOWN 2.3283064365386963e-10f    // 2^-32, of their sums

// v = h + m + l exactly (finite v, 0 or from 2^-110).
__device__ __forceinline__ void fbc_f3_split2(float v0, float v1, fbc_u32& h, fbc_u32& m, fbc_u32& l) {
    h = fbc_pack_bf16x2(v0, v1);
    const float r0 = v0 - __uint_as_float(h << 16), r1 = v1 - __uint_as_float(h & 0xFFFF0000u);
    m = fbc_pack_bf16x2(r0, r1);
    l = fbc_pack_bf16x2(r0 - __uint_as_float(m << 16), r1 - __uint_as_float(m & 0xFFFF0000u));
}

__device__ __forceinline__ void fbc_f3_split4(const float (&v)[4], fbc_u32 (&h)[2], fbc_u32 (&m)[2], fbc_u32 (&l)[2]) {
    fbc_f3_split2(v[0], v[1], h[0], m[0], l[0]);
    fbc_f3_split2(v[2], v[3], h[1], m[1], l[1]);
}

// Packed multiplies: with scalar ones the dense 512x512x32 * 256x5x5 took 429 us
// instead of 425.
template <int N>
__device__ __forceinline__ void fbc_f3_scale(float (&v)[N], float s) {
#pragma unroll
    for (int k = 0; k < N; k += 2)
        asm("{\n .reg .b64 t, u;\n mov.b64 t, {%0, %1};\n mov.b64 u, {%2, %2};\n mul.rn.f32x2 t, t, u;\n"
            " mov.b64 {%0, %1}, t;\n}\n" : "+f"(v[k]), "+f"(v[k + 1]) : "f"(s));
}

// FP32 operands into the split's range; the BF16 modes take them as they are.
template <int ORD, int N>
__device__ __forceinline__ void fbc_f3_up(float (&v)[N]) {
    if constexpr (ORD == 3) fbc_f3_scale(v, FBC_F3_UP);
}

// The first ORD orders of one chunk (8 values) to shared memory, `ord` bytes apart.
template <int ORD = 3>
__device__ __forceinline__ void fbc_f3_put(const float (&v)[8], fbc_u32 dst, fbc_u32 ord) {
    fbc_u32 h[4], m[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) fbc_f3_split2(v[2 * k], v[2 * k + 1], h[k], m[k], l[k]);
    fbc_st_shared_v4(dst, h[0], h[1], h[2], h[3]);
    if (ORD > 1) fbc_st_shared_v4(dst + ord, m[0], m[1], m[2], m[3]);
    if (ORD > 2) fbc_st_shared_v4(dst + 2 * ord, l[0], l[1], l[2], l[3]);
}

template <int ORD = 3>
__device__ __forceinline__ void fbc_f3_put(const float (&v)[4], fbc_u32 dst, fbc_u32 ord) {
    fbc_u32 h[2], m[2], l[2];
    fbc_f3_split4(v, h, m, l);
    fbc_st_shared_v2(dst, h[0], h[1]);
    if (ORD > 1) fbc_st_shared_v2(dst + ord, m[0], m[1]);
    if (ORD > 2) fbc_st_shared_v2(dst + 2 * ord, l[0], l[1]);
}

__device__ __forceinline__ int fbc_f3_row(int v, const FbcF3Params& P) {
    return P.vw == 1 ? v : (int)(__umulhi((unsigned)v, P.vw_mul) >> P.vw_shift);
}

template <class G>
__device__ __forceinline__ float fbc_f3_masked(float v, const float* m, const FbcF3Params& P) {
    if constexpr (G::MASK) {
        const float t = __ldg(m);
        return (t > P.lo && t < P.hi) ? v : 0.f;
    }
    return v;
}

// The epilogue and store of 8 consecutive columns col0 .. col0 + 7 of the tile
// at output pixel (row group pg, column q); n0 = first filter of the tile.
template <class G>
__device__ __forceinline__ void fbc_f3_store8(const FbcF3Params& P, int pg, int q, int n0, int col0, float (&v)[8]) {
    if constexpr (G::EPI == 1) {
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = fminf(fmaxf(v[k], P.lo), P.hi);
    }
    if constexpr (G::EPI == 2) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            v[k] = fbc_user_epi(v[k], G::R > 1 ? (col0 + k) % G::NF : n0 + col0 + k, P.lo, P.hi);
    }
    // group size of contiguous, equally aligned filters of one output row
    constexpr int GS = G::NF % 8 == 0 ? 8 : G::NF % 4 == 0 ? 4 : 1;
#pragma unroll
    for (int g = 0; g < 8; g += GS) {
        const int col = col0 + g;
        const int r = G::R > 1 ? col / G::NF : 0;
        const int n = G::R > 1 ? col - r * G::NF : n0 + col;
        const int p = pg * G::R + r;
        if (r >= G::R || p >= P.out_h || n >= G::NF) continue;
        float* dst = P.y + ((long long)p * P.out_w + q) * G::NF + n;
        if constexpr (GS == 8) {
            if ((reinterpret_cast<unsigned long long>(P.y) & 31) == 0) {
                asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]),
                             "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                             : "memory");
            } else {
                *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4*>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
            }
        } else if constexpr (GS == 4) {
            *reinterpret_cast<float4*>(dst) = make_float4(v[g], v[g + 1], v[g + 2], v[g + 3]);
        } else {
            dst[0] = v[g];
        }
    }
}

__device__ __forceinline__ float fbc_f3_bf16(float v) { return __uint_as_float(fbc_pack_bf16x2(v, 0.f) << 16); }

// x w added to acc in FP32 (the BF16 modes: the products of the rounded values).
template <class G>
__device__ __forceinline__ float fbc_f3_mac(float x, float w, float acc) {
    if constexpr (G::ORD == 3) return fmaf(x, w, acc);
    const float xh = fbc_f3_bf16(x), wh = fbc_f3_bf16(w);
    if constexpr (G::ORD == 2) {
        acc = fmaf(xh, fbc_f3_bf16(w - wh), acc);
        acc = fmaf(fbc_f3_bf16(x - xh), wh, acc);
    }
    return fmaf(xh, wh, acc);
}

// N consecutive floats (N = 4: on a 16-byte boundary).
template <int N>
__device__ __forceinline__ void fbc_f3_ldg(const float* p, float (&v)[N]) {
    if constexpr (N == 4) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = f.x;
        v[1] = f.y;
        v[2] = f.z;
        v[3] = f.w;
    } else {
        v[0] = __ldg(p);
    }
}

// Columns col0 .. col0 + 7 of those of the warp's 32 pixels that `mask` names, again,
// with FP32 FMAs from global memory.  Bound by the loads: four lanes share the FW C
// products of a filter row (consecutive floats of x, and of an unflipped bank) and
// hold four pixels x 8 columns each, so that 12 loads of 16 bytes feed 128 FMAs, with
// 8 pixels' lines per load of x and one per load of w.  512x512x32 * 256x5x5 with one
// NaN pixel 0.43 ms, one NaN weight 0.53, NaN all over the image 4.5 (one thread per
// pixel and whole tiles: 12, 63 and 304; without NaN 0.40; the FMA kernel 1.93).
template <class G>
__device__ __forceinline__ void fbc_f3_redo(const FbcF3Params& P, fbc_u32 mask, int pg, int q, int n0, int col0) {
    if (G::R == 1 ? n0 + col0 >= G::NF : col0 >= G::R * G::NF) return;
    constexpr int V = G::VA ? 4 : 1;
    const int part = threadIdx.x & 3, slot = (threadIdx.x & 31) >> 2;
    int row0[4], col[4];
    bool on[4];
    float acc[4][8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        row0[t] = __shfl_sync(0xFFFFFFFFu, pg, 8 * t + slot) * G::R - P.pad_y;
        col[t] = __shfl_sync(0xFFFFFFFFu, q, 8 * t + slot) - P.pad_x;
        on[t] = (mask >> (8 * t + slot)) & 1u;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[t][k] = 0.f;
    }
    const int r0 = G::R > 1 ? col0 / G::NF : 0, r1 = G::R > 1 ? min(G::R - 1, (col0 + 7) / G::NF) : 0;
#pragma unroll 1
    for (int ri = 0; ri < (r1 - r0 + 1) * G::FH; ++ri) {
        const int r = r0 + ri / G::FH, i = ri % G::FH;
        const int nb = G::R > 1 ? col0 - r * G::NF : n0 + col0;     // filter of the first column
#pragma unroll 1
        for (int e0 = part * V; e0 < G::FW * G::C; e0 += 4 * V) {
            const int j = e0 / G::C, c = e0 % G::C;
            // every load before the first FMA, none behind a branch: what takes no part
            // reads the first pixel or a neighbouring filter and is left out of the sums
            float xv[4][V], wv[8][V];
            bool ok[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int xr = row0[t] + r + i, xc = col[t] + j;
                ok[t] = on[t] && xr >= 0 && xr < P.in_h && xc >= 0 && xc < P.in_w;
                const unsigned o = ok[t] ? ((unsigned)xr * P.in_w + xc) * G::C + c : 0u;
                fbc_f3_ldg<V>(P.x + o, xv[t]);
                if constexpr (G::MASK) {
                    float mv[V];
                    fbc_f3_ldg<V>(P.m + o, mv);
#pragma unroll
                    for (int e = 0; e < V; ++e) xv[t][e] = mv[e] > P.lo && mv[e] < P.hi ? xv[t][e] : 0.f;
                }
            }
            if constexpr (G::FLIP && G::NF % 4 == 0) {
#pragma unroll
                for (int k = 0; k < 8; k += 4) {
                    const int n = min(max(nb + k, 0), G::NF - 4);
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        float f[4];
                        fbc_f3_ldg<4>(P.w + (((unsigned)(c + e) * G::FH + (G::FH - 1 - i)) * G::FW + (G::FW - 1 - j)) * G::NF + n, f);
#pragma unroll
                        for (int h = 0; h < 4; ++h) wv[k + h][e] = f[h];
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int n = min(max(nb + k, 0), G::NF - 1);
                    if constexpr (!G::FLIP) {
                        fbc_f3_ldg<V>(P.w + ((unsigned)n * G::FH + i) * (G::FW * G::C) + e0, wv[k]);
                    } else {
#pragma unroll
                        for (int e = 0; e < V; ++e)
                            fbc_f3_ldg<1>(P.w + (((unsigned)(c + e) * G::FH + (G::FH - 1 - i)) * G::FW + (G::FW - 1 - j)) * G::NF + n,
                                          reinterpret_cast<float(&)[1]>(wv[k][e]));
                    }
                }
            }
            // a tap outside the image takes no part (it could be 0 x inf); without a border there is none
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (G::R == 1 || (nb + k >= 0 && nb + k < G::NF)) {
#pragma unroll
                    for (int t = 0; t < 4; ++t)
#pragma unroll
                        for (int e = 0; e < V; ++e)
                            if (!G::FLIP || ok[t]) acc[t][k] = fbc_f3_mac<G>(xv[t][e], wv[k][e], acc[t][k]);
                }
        }
    }
    // the four lanes' sums; each stores one of the four pixels
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            acc[t][k] += __shfl_xor_sync(0xFFFFFFFFu, acc[t][k], 1);
            acc[t][k] += __shfl_xor_sync(0xFFFFFFFFu, acc[t][k], 2);
        }
        v[k] = part == 0 ? acc[0][k] : part == 1 ? acc[1][k] : part == 2 ? acc[2][k] : acc[3][k];
    }
    const int src = 8 * part + slot;
    pg = __shfl_sync(0xFFFFFFFFu, pg, src);
    q = __shfl_sync(0xFFFFFFFFu, q, src);
    if ((mask >> src) & 1u) fbc_f3_store8<G>(P, pg, q, n0, col0, v);
}

// A note: the CTA's item and the accumulating warp (low 3 bits) that met non-finite sums,
// and for each group of 8 columns which of its four groups of 8 pixels hold them.
struct FbcF3Note {
    fbc_u32 where, what;
};
#define FBC_F3_NOTES 120     // with the rest at most 1 KB of static shared memory

// Position in a CTA's sequence of (work item, unit); item = filter tile * mtiles + pixel tile.
template <class G>
struct FbcF3Pos {
    int item, u, mt, ft;       // mt, ft: the item's pixel and filter tile, kept without a division
    __device__ __forceinline__ void wrap(const FbcF3Params& P) {
        while (mt >= P.mtiles) {
            mt -= P.mtiles;
            ++ft;
        }
    }
    __device__ __forceinline__ void start(const FbcF3Params& P) {
        item = mt = blockIdx.x;
        u = ft = 0;
        wrap(P);
    }
    __device__ __forceinline__ bool valid(const FbcF3Params& P) const { return item < P.nitems; }
    __device__ __forceinline__ void next(const FbcF3Params& P) {
        if (++u < G::NU) return;
        u = 0;
        item += gridDim.x;
        mt += gridDim.x;
        wrap(P);
    }
};

// Item `it` of unit j: slab row it / (NPX QA) of the unit, a quad (VA) or a chunk
// of 8 of one of its pixels.
template <class G>
__device__ __forceinline__ void fbc_f3_a_item(int it, int& k, int& px, int& sub) {
    k = G::RU > 1 ? it / (G::NPX * G::QA) : 0;
    const int r = it - k * (G::NPX * G::QA);
    px = G::VA ? r / G::QA : r % G::NPX;
    sub = G::VA ? r % G::QA : r / G::NPX;
}

template <class G>
__device__ __forceinline__ void fbc_f3_load_a(const FbcF3Params& P, const FbcF3Pos<G>& j, int it, float (&v)[G::WA],
                                              float (&mv)[G::LATE ? G::WA : 1]) {
    const int cg = G::channel_group(j.u);
    int k, px, sub;
    fbc_f3_a_item<G>(it, k, px, sub);
    const int ri = G::row0(j.u) + k;
    const int vp = j.mt * 128 + G::tap_group(j.u) * G::JT + px;
#pragma unroll
    for (int e = 0; e < G::WA; ++e) v[e] = 0.f;
    if constexpr (G::VA && G::R == 1 && !G::FLIP) {
        // no border and one row per tile row: the slab is a run of x itself (past a row's
        // end it reads the next row, for outputs that are dropped and taps that are zero)
        const int pix = vp + ri * P.in_w;
        const int ch = G::PP == 1 ? cg * G::GC + sub * 4 : 0;
        if (it >= G::NIT || ri >= G::ROWS || pix >= P.in_h * P.in_w || ch >= G::C) return;
        const float4 f = __ldg(reinterpret_cast<const float4*>(P.x + (unsigned)(pix * G::C + ch)));
        v[0] = f.x;
        v[1] = f.y;
        v[2] = f.z;
        v[3] = f.w;
        return;
    }
    const int pg = fbc_f3_row(vp, P);
    const int col = vp - pg * P.vw - P.pad_x;
    const int row = pg * G::R + ri - P.pad_y;
    if (it >= G::NIT || ri >= G::ROWS || row < 0 || row >= P.in_h) return;
    if constexpr (G::VA) {
        const int ch = cg * G::GC + sub * 4;
        if (col < 0 || col >= P.in_w || (G::PP == 1 && ch >= G::C)) return;
        const unsigned o = (unsigned)((row * P.in_w + col) * G::C + (G::PP == 1 ? ch : 0));
        const float4 f = __ldg(reinterpret_cast<const float4*>(P.x + o));
        v[0] = f.x;
        v[1] = f.y;
        v[2] = f.z;
        v[3] = f.w;
        if constexpr (G::LATE) {
            const float4 g = __ldg(reinterpret_cast<const float4*>(P.m + o));
            mv[0] = g.x;
            mv[1] = g.y;
            mv[2] = g.z;
            mv[3] = g.w;
        } else if constexpr (G::MASK) {
            const float4 g = __ldg(reinterpret_cast<const float4*>(P.m + o));
            if (!(g.x > P.lo && g.x < P.hi)) v[0] = 0.f;
            if (!(g.y > P.lo && g.y < P.hi)) v[1] = 0.f;
            if (!(g.z > P.lo && g.z < P.hi)) v[2] = 0.f;
            if (!(g.w > P.lo && g.w < P.hi)) v[3] = 0.f;
        }
    } else {
        const int ch = G::PP == 1 ? cg * G::GC + sub * 8 : 0;
#pragma unroll
        for (int e = 0; e < G::WA; ++e) {
            const int cc = col + e / G::CP, c = ch + e % G::CP;
            if (cc < 0 || cc >= P.in_w || c >= G::C) continue;
            const unsigned o = (unsigned)((row * P.in_w + cc) * G::C + c);
            if constexpr (G::LATE) {
                v[e] = __ldg(P.x + o);
                mv[e] = __ldg(P.m + o);
            } else {
                v[e] = fbc_f3_masked<G>(__ldg(P.x + o), P.m + o, P);
            }
        }
    }
}

// Item `it` of a unit into the A slot at dst; `all`: every thread has one in this pass
// (no branch: the conversions of several passes interleave).
template <class G>
__device__ __forceinline__ void fbc_f3_put_a(const FbcF3Params& P, int it, bool all, float (&v)[G::WA],
                                             const float (&mv)[G::LATE ? G::WA : 1], fbc_u32 dst) {
    if (!all && it >= G::NIT) return;
    if constexpr (G::LATE) {
#pragma unroll
        for (int e = 0; e < G::WA; ++e)
            if (!(mv[e] > P.lo && mv[e] < P.hi)) v[e] = 0.f;
    }
    fbc_f3_up<G::ORD>(v);
    int k, px, sub;
    fbc_f3_a_item<G>(it, k, px, sub);
    const fbc_u32 d = dst + (fbc_u32)k * G::SLAB + (fbc_u32)px * 16u;
    if constexpr (!G::VA) {
        fbc_f3_put<G::ORD>(v, d + (fbc_u32)sub * G::PLANE, G::AORD);
    } else if constexpr (G::PP == 2) {
        // a pixel of 4 channels: first half of chunk px and second half of chunk px - 1
        fbc_u32 h[2], m[2], l[2];
        fbc_f3_split4(v, h, m, l);
        if (px < G::LS) {
            fbc_st_shared_v2(d, h[0], h[1]);
            if (G::ORD > 1) fbc_st_shared_v2(d + G::AORD, m[0], m[1]);
            if (G::ORD > 2) fbc_st_shared_v2(d + 2 * G::AORD, l[0], l[1]);
        }
        if (px > 0) {
            fbc_st_shared_v2(d - 8u, h[0], h[1]);
            if (G::ORD > 1) fbc_st_shared_v2(d - 8u + G::AORD, m[0], m[1]);
            if (G::ORD > 2) fbc_st_shared_v2(d - 8u + 2 * G::AORD, l[0], l[1]);
        }
    } else {
        fbc_f3_put<G::ORD>(v, d + (fbc_u32)(sub >> 1) * G::PLANE + (fbc_u32)(sub & 1) * 8u, G::AORD);
    }
}

// The bank split: block (b, filter tile) splits chunks 256 b .. of the tile's
// NU x NBC chunks (unit, slab row, step, half, column), one per thread, columns
// fastest, into the B stage images.
template <class G>
__device__ __forceinline__ void fbc_f32tc_bank_body(const FbcF3Params& P) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int id = blockIdx.x * FBC_F3_BANK_THREADS + threadIdx.x;
    if (id < G::NU * G::NBC) {
        const int u = id / G::NBC, it = id % G::NBC;
        const int col = it % G::NT, kq = (it / G::NT) % (2 * G::S), ri = G::row0(u) + it / (G::NT * 2 * G::S);
        const int r = G::R > 1 ? col / G::NF : 0;
        const int n = G::R > 1 ? col - r * G::NF : (int)blockIdx.y * G::NT + col;
        const int i = ri - r;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0.f;
        if (r < G::R && n < G::NF && i >= 0 && i < G::FH) {
            const int jl = G::PACK ? kq * G::PP : kq / G::PL;     // first tap of the chunk in its group
            const int ch = G::PP > 1 ? 0 : G::PACK ? G::channel_group(u) * 8 : G::channel_group(u) * G::GC + (kq % G::PL) * 8;
            const int tap = G::tap_group(u) * G::JT + jl;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int dt = e / G::CP, c = ch + e % G::CP;
                if (jl + dt >= G::JT || tap + dt >= G::FW || c >= G::C) continue;
                const unsigned o =
                    G::FLIP ? (unsigned)(((c * G::FH + (G::FH - 1 - i)) * G::FW + (G::FW - 1 - tap - dt)) * G::NF + n)
                            : (unsigned)(((n * G::FH + i) * G::FW + tap + dt) * G::C + c);
                v[e] = __ldg(P.w + o);
            }
        }
        fbc_f3_up<G::ORD>(v);
        fbc_u32 h[4], m[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) fbc_f3_split2(v[2 * k], v[2 * k + 1], h[k], m[k], l[k]);
        unsigned char* dst = P.bank + ((long long)blockIdx.y * G::NU + u) * G::BUNIT + (it / G::NT) * G::BCH + col * 16;
        *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
        if (G::ORD > 1) *reinterpret_cast<uint4*>(dst + G::NT * 16) = make_uint4(m[0], m[1], m[2], m[3]);
        if (G::ORD > 2) *reinterpret_cast<uint4*>(dst + 2 * G::NT * 16) = make_uint4(l[0], l[1], l[2], l[3]);
    }
}

// The noted outputs of a CTA, by every one of its warps; the items from `from` on, for
// which there was no room, whole.  Not inlined: inlined, or noted group by group, it cost
// the pipeline registers (512x512x32 * 256x5x5 401 instead of 392 us, split BF16
// 256x256x8 * 64x9x9 24.2 either way, BF16 2048x2048x4 * 4x8x8 62.4 instead of 61.3).
template <class G>
__device__ __noinline__ void fbc_f3_redo_noted(const FbcF3Params& P0, const FbcF3Note* list, int noted, int from) {
    const FbcF3Params P = P0;     // in registers: by reference it took half as long again
    constexpr int NG = G::NT / 16;
    const int lane = threadIdx.x & 31;
    const int items = (P.nitems - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const int listed = min(noted, FBC_F3_NOTES);
    const int count = listed + (from < items ? (items - from) * 8 : 0);
    // a group of all notes after the other: one bad filter is work for every warp
    int g = 0, e = threadIdx.x >> 5;
#pragma unroll 1
    for (;; e += FBC_F3_THREADS / 32) {
        for (; e >= count && g < NG; ++g) e -= count;
        if (g >= NG) break;
        // beyond the list: every warp's part of an item
        const fbc_u32 where = e < listed ? list[e].where : (fbc_u32)(from * 8 + e - listed);
        const fbc_u32 bytes = e < listed ? list[e].what >> (4 * g) & 0xFu : 0xFu;
        if (bytes == 0) continue;
        const int item = (int)(blockIdx.x + (where >> 3) * gridDim.x), wq = (int)where & 7;
        const int v = (item % P.mtiles) * 128 + (wq & 3) * 32 + lane;
        const int pg = fbc_f3_row(v, P), q = v - pg * P.vw;
        const bool inside = q < P.out_w && pg * G::R < P.out_h && ((bytes >> (lane >> 3)) & 1u);
        const fbc_u32 mask = __ballot_sync(0xFFFFFFFFu, inside);
        fbc_f3_redo<G>(P, mask, pg, q, G::R > 1 ? 0 : item / P.mtiles * G::NT, (wq >> 2) * (G::NT / 2) + 8 * g);
    }
}

template <class G>
__device__ __forceinline__ void fbc_f32tc_body(const FbcF3Params& P) {
    __shared__ int s_abort;
    __shared__ fbc_u32 s_tmem;
    __shared__ FbcF3Note s_bad[FBC_F3_NOTES];   // where sums were not finite, and how often that was noted
    __shared__ int s_nbad, s_bad_from;          // (from item s_bad_from on there was no room)
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const fbc_u32 sbase = fbc_smem_addr(fbc_tc_smem);
    // barrier table: a_full[na] a_empty[na] b_full[2][nb] b_empty[2][nb] acc_full[2] acc_empty[2] drain[2]
    const fbc_u32 a_full0 = sbase + P.bar_off;
    const fbc_u32 a_empty0 = a_full0 + 8u * P.na;
    const fbc_u32 b_full0 = a_empty0 + 8u * P.na;
    const fbc_u32 b_empty0 = b_full0 + 16u * P.nb;
    const fbc_u32 acc_full0 = b_empty0 + 16u * P.nb;
    const fbc_u32 acc_empty0 = acc_full0 + 16u;
    const fbc_u32 drain_bar = acc_empty0 + 16u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < P.na; ++s) {
            fbc_mbar_init(a_full0 + 8u * s, FBC_F3_CONV_WARPS);
            fbc_mbar_init(a_empty0 + 8u * s, 1);
        }
        for (int s = 0; s < 2 * P.nb; ++s) {
            fbc_mbar_init(b_full0 + 8u * s, 1);
            fbc_mbar_init(b_empty0 + 8u * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            fbc_mbar_init(acc_full0 + 8u * s, 2);    // the MMA commit, and the issuing thread itself
            fbc_mbar_init(acc_empty0 + 8u * s, FBC_F3_EPI_WARPS);
        }
        fbc_mbar_init(drain_bar, 1);
        fbc_mbar_init(drain_bar + 8u, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        s_nbad = 0;
        s_bad_from = 0x7FFFFFFF;
    }
    if (warp == 15) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(fbc_smem_addr(&s_tmem)),
                     "n"(G::TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fbc_tc_fence_before();
    __syncthreads();
    fbc_tc_fence_after();
    const fbc_u32 tmem = s_tmem;
    volatile int* abort_flag = &s_abort;
    // launched as a programmatic dependent: the previous kernel of the stream is
    // complete and visible before anything below touches global memory
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp >= 8 && warp < 8 + FBC_F3_CONV_WARPS) {
        // ------------------------------------------------------------ converters
        const int ct = threadIdx.x - 8 * 32;
        FbcF3Pos<G> ja, jn;      // unit being written, unit being loaded
        ja.start(P);
        jn = ja;
        float abuf[G::PA][G::KA][G::WA], mbuf[G::PA][G::KA][G::LATE ? G::WA : 1];
        auto load_a = [&](float (&buf)[G::KA][G::WA], float (&mask)[G::KA][G::LATE ? G::WA : 1]) {
            if (!jn.valid(P)) return;
#pragma unroll
            for (int k = 0; k < G::KA; ++k) fbc_f3_load_a<G>(P, jn, ct + k * G::NCT, buf[k], mask[k]);
            jn.next(P);
        };
#pragma unroll
        for (int s = 0; s < G::PA; ++s) load_a(abuf[s], mbuf[s]);
        int as = 0;
        fbc_u32 aph = 0;
        bool ok = true;
        while (ok && ja.valid(P)) {
#pragma unroll
            for (int s = 0; s < G::PA; ++s) {
                if (!ok || !ja.valid(P)) break;
                if (!(ok = fbc_wait(a_empty0 + 8u * as, aph ^ 1, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                const fbc_u32 dst = sbase + (fbc_u32)as * G::ASLOT;
#pragma unroll
                for (int k = 0; k < G::KA; ++k)
                    fbc_f3_put_a<G>(P, ct + k * G::NCT, (k + 1) * G::NCT <= G::NIT, abuf[s][k], mbuf[s][k], dst);
                fbc_fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) fbc_mbar_arrive(a_full0 + 8u * as);
                if (++as == P.na) { as = 0; aph ^= 1; }
                load_a(abuf[s], mbuf[s]);
                ja.next(P);
            }
        }
    } else if (warp == 13) {
        if (lane == 0) {
            // -------------------------------------------------------- bank producer
            // both rings in turn, whichever has a free stage
            struct {
                FbcF3Pos<G> j;
                int st, bs;
                fbc_u32 ph, it;
            } q[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                q[r].j.start(P);
                if (r == 1) q[r].j.next(P);
                q[r].st = q[r].bs = 0;
                q[r].ph = q[r].it = 0;
            }
            fbc_u64 t0 = fbc_globaltimer();
            fbc_u32 idle = 0;
            bool ok = true;
            while (ok && (q[0].j.valid(P) || q[1].j.valid(P))) {
                bool moved = false;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (!q[r].j.valid(P)) continue;
                    const int slot = r * P.nb + q[r].bs;
                    if (!fbc_mbar_test(b_empty0 + 8u * slot, q[r].ph ^ 1)) continue;
                    moved = true;
                    const fbc_u32 off = (fbc_u32)q[r].st * G::BSTAGE;
                    const fbc_u32 bytes = min(G::BSTAGE, G::BUNIT - off);
                    fbc_mbar_expect_tx(b_full0 + 8u * slot, bytes);
                    if (!FBC_F3_DROP || r > 0 || q[r].it > 0)
                        fbc_bulk_g2s(sbase + P.b_off + (fbc_u32)slot * G::BSTAGE,
                                     P.bank + ((long long)q[r].j.ft * G::NU + q[r].j.u) * G::BUNIT + off, bytes,
                                     b_full0 + 8u * slot);
                    ++q[r].it;
                    if (++q[r].bs == P.nb) { q[r].bs = 0; q[r].ph ^= 1; }
                    if (++q[r].st == G::NST) {
                        q[r].st = 0;
                        q[r].j.next(P);
                        q[r].j.next(P);
                    }
                }
                if (moved) {
                    idle = 0;
                } else if ((++idle & 63u) == 0) {
                    // nothing freed for a while: stop with the CTA, or after the bound
                    if (idle == 64u) t0 = fbc_globaltimer();
                    if (*abort_flag) ok = false;
                    if (fbc_globaltimer() - t0 > P.wait_ns) {
                        *abort_flag = 1;
                        *(volatile int*)P.err = FBC_F3_ERR_WAIT;
                        __threadfence_system();
                        ok = false;
                    }
                }
            }
            if (!ok) {
                // wait (bounded) for the copies still in flight into the rings
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const fbc_u32 k0 = q[r].it > (fbc_u32)P.nb ? q[r].it - P.nb : 0;
                    for (fbc_u32 k = k0; k < q[r].it; ++k)
                        fbc_wait_drain(b_full0 + 8u * (r * P.nb + k % P.nb), (k / P.nb) & 1, P);
                }
            }
        }
    } else if (warp >= 14) {
        if (lane == 0) {
            // -------------------------------------------------------- MMA issuers
            // Issuing one MMA takes a thread 40 to 60 cycles, a barrier wait or a commit
            // about 70; at 32 to 96 cycles per MMA one thread alone left the tensor core
            // idle a third of the time (dense 512 x 512 x 32 * 256 x 5 x 5: 0.43 ms).
            const fbc_u32 idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);   // FP32 += BF16 x BF16, M = 128
            const fbc_u32 id3 = idesc0 | ((3u * G::NT >> 3) << 17);
            const fbc_u32 id2 = idesc0 | ((2u * G::NT >> 3) << 17);
            const fbc_u32 id1 = idesc0 | ((1u * G::NT >> 3) << 17);
            const fbc_u32 idn[3] = {G::ORD == 3 ? id3 : G::ORD == 2 ? id2 : id1, G::ORD == 3 ? id2 : id1, id1};
            // descriptors: the start address (16-byte units) sits in the low bits of the
            // low word and never carries out of its field; the high word is constant
            const fbc_u64 adesc0 = fbc_smem_desc(sbase, G::PACK ? 16u * G::PP : G::PLANE, 128);
            const fbc_u32 ring = (fbc_u32)(warp - 14) * P.nb;      // this thread's B stages
            const fbc_u64 bdesc0 = fbc_smem_desc(sbase + P.b_off + ring * G::BSTAGE, G::BCH, 128);
            const fbc_u32 ahi = (fbc_u32)(adesc0 >> 32), bhi = (fbc_u32)(bdesc0 >> 32);
            const int acc = warp - 14;         // this thread's accumulator set
            const fbc_u32 d = tmem + (fbc_u32)(acc * G::ORD * G::NT);
            int as = 0, bs = 0;
            fbc_u32 aph = 0, bph = 0, accph = 0;
            int turn = 0;
            bool ok = true, issued = false;
            FbcF3Pos<G> j;
            for (j.start(P); j.valid(P); j.next(P), turn ^= 1) {
                if (turn == acc) {
                    if (!(ok = fbc_wait(acc_empty0 + 8u * acc, accph ^ 1, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                    if (!(ok = fbc_wait(a_full0 + 8u * as, aph, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                    accph ^= 1;
                    const fbc_u32 alo = (fbc_u32)adesc0 + ((fbc_u32)as * G::ASLOT >> 4);
                    const int steps = min(G::RU, G::ROWS - G::row0(j.u)) * G::S;   // the last unit may hold fewer rows
#pragma unroll
                    for (int st = 0; st < G::NST; ++st) {
                        if (!(ok = fbc_wait(b_full0 + 8u * (ring + bs), bph, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                        fbc_tc_fence_after();
                        issued = true;
                        const fbc_u32 blo = (fbc_u32)bdesc0 + ((fbc_u32)bs * G::BSTAGE >> 4);
#pragma unroll
                        for (int q = 0; q < G::BS; ++q) {
                            const int e = st * G::BS + q, k = e / G::S, s = e % G::S;
                            if (e >= G::STEPS || (G::ROWS % G::RU != 0 && k > 0 && e >= steps)) break;
                            const fbc_u32 ao = k * G::SLAB + (G::PACK ? 2u * s * G::PP * 16u
                                                                      : (s % (G::GC / 16)) * 2u * G::PLANE + (s / (G::GC / 16)) * 16u);
                            const fbc_u32 a1 = alo + (ao >> 4), b = blo + (q * G::BSTEP >> 4);
                            // order o of x with the first ORD - o of w
                            fbc_umma_lo(d, a1, ahi, b, bhi, idn[0], e > 0 ? 1u : 0u);
                            if constexpr (G::ORD > 1) fbc_umma_lo(d + G::NT, a1 + (G::AORD >> 4), ahi, b, bhi, idn[1], 1u);
                            if constexpr (G::ORD > 2)
                                fbc_umma_lo(d + 2 * G::NT, a1 + (2 * G::AORD >> 4), ahi, b, bhi, idn[2], 1u);
                        }
                        fbc_umma_commit<1>(b_empty0 + 8u * (ring + bs));
                        if (++bs == P.nb) { bs = 0; bph ^= 1; }
                    }
                    if (!ok) break;
                    fbc_umma_commit<1>(a_empty0 + 8u * as);
                    fbc_umma_commit<1>(acc_full0 + 8u * acc);
                    fbc_mbar_arrive(acc_full0 + 8u * acc);   // this thread has seen the converters' writes
                }
                if (++as == P.na) { as = 0; aph ^= 1; }
            }
            if (!ok && issued) {
                fbc_umma_commit<1>(drain_bar + 8u * acc);
                fbc_wait_drain(drain_bar + 8u * acc, 0, P);
            }
        }
    } else {
        // ------------------------------------------------------------ accumulate and store
        constexpr int HC = G::NT / 2;          // columns of this warp
        const int lq = warp & 3, half = warp >> 2;
        const fbc_u32 trow = tmem + ((fbc_u32)(lq * 32) << 16) + (fbc_u32)(half * HC);
        int acc = 0, ord = 0;
        fbc_u32 accph = 0;
        bool ok = true;
        // A finished tile is stored in pieces between the drains of the next one: storing
        // it at once held both accumulator sets, and with them the tensor core, for a
        // tenth of the time.
        constexpr int NG = HC / 8, PER = (NG + G::NU - 1) / G::NU;    // groups of 8 columns, groups per drain
        float out[HC];
        int o_pg = 0, o_q = 0, o_n0 = 0, o_next = NG;
        auto store_some = [&](int count) {
#pragma unroll
            for (int g = 0; g < NG; ++g)
                if (g >= o_next && g < o_next + count) {
                    float v8[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v8[e] = out[8 * g + e];
                    fbc_f3_store8<G>(P, o_pg, o_q, o_n0, half * HC + 8 * g, v8);
                }
            o_next += count;
        };
        for (int item = blockIdx.x; item < P.nitems && ok; item += gridDim.x, ++ord) {
            const int mt = item % P.mtiles;
            const int n0 = G::R > 1 ? 0 : (item / P.mtiles) * G::NT;
            float sum[HC];
#pragma unroll
            for (int k = 0; k < HC; ++k) sum[k] = 0.f;
            for (int u = 0; u < G::NU; ++u) {
                if (!(ok = fbc_wait(acc_full0 + 8u * acc, accph, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                fbc_tc_fence_after();
                const fbc_u32 ta = trow + (fbc_u32)(acc * G::ORD * G::NT);
#pragma unroll
                for (int k = 0; k < HC; k += 8) {
                    fbc_u32 r0[8], r1[8], r2[8];
                    fbc_tmem_ld32x32b_x8_async(ta + k, r0);
                    if constexpr (G::ORD > 1) fbc_tmem_ld32x32b_x8_async(ta + G::NT + k, r1);
                    if constexpr (G::ORD > 2) fbc_tmem_ld32x32b_x8_async(ta + 2 * G::NT + k, r2);
                    fbc_tmem_ld_wait();
                    fbc_reg_fence8(r0);
                    if constexpr (G::ORD > 1) fbc_reg_fence8(r1);
                    if constexpr (G::ORD > 2) fbc_reg_fence8(r2);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float s = __uint_as_float(r0[e]);
                        if constexpr (G::ORD == 2) s += __uint_as_float(r1[e]);
                        if constexpr (G::ORD == 3) s += __uint_as_float(r1[e]) + __uint_as_float(r2[e]);
                        sum[k + e] += s;
                    }
                }
                fbc_tc_fence_before();
                __syncwarp();
                if (lane == 0) fbc_mbar_arrive(acc_empty0 + 8u * acc);
                acc ^= 1;
                if (acc == 0) accph ^= 1;
                if (o_next < NG) store_some(PER);
            }
            if (!ok) break;
            // the tile is complete
            const int v = mt * 128 + lq * 32 + lane;
            o_pg = fbc_f3_row(v, P);
            o_q = v - o_pg * P.vw;
            o_n0 = n0;
            const bool inside = o_q < P.out_w && o_pg * G::R < P.out_h;
            // a sum is finite unless its difference with itself is not zero
            float z = 0.f;
#pragma unroll
            for (int k = 0; k < HC; ++k) {
                z += sum[k] - sum[k];
                out[k] = G::ORD == 3 ? sum[k] * FBC_F3_DOWN : sum[k];
            }
            if (__any_sync(0xFFFFFFFFu, inside && !(z == 0.f))) {
                fbc_u32 bad = 0;
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    z = 0.f;
#pragma unroll
                    for (int k = 8 * g; k < 8 * g + 8; ++k) z += out[k] - out[k];
                    bad |= inside && !(z == 0.f) ? 1u << (4 * g) : 0u;
                }
                bad = __reduce_or_sync(0xFFFFFFFFu, bad << (lane >> 3));
                if (lane == 0) {
                    const int k = atomicAdd(&s_nbad, 1);
                    if (k < FBC_F3_NOTES) s_bad[k] = FbcF3Note{(fbc_u32)ord << 3 | (fbc_u32)warp, bad};
                    else atomicMin(&s_bad_from, ord);
                }
            }
            o_next = inside ? 0 : NG;
            __syncwarp();
        }
        if (o_next < NG) store_some(NG);
    }
    __syncwarp();
    fbc_tc_fence_before();
    __syncthreads();
    fbc_tc_fence_after();
    if (warp == 15)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(G::TMEM));
    // the noted groups: the stores above came before the barrier
    if (s_nbad > 0 && s_abort == 0) fbc_f3_redo_noted<G>(P, s_bad, s_nbad, s_bad_from);
}

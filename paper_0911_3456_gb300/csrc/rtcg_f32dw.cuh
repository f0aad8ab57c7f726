// rtcg_f32dw.cuh -- dL/dw in FP32 on the tensor cores, compiled at plan time by
// NVRTC for sm_103a.  Embedded as a string and placed after rtcg_f32tc.cuh, whose
// three-way BF16 split it shares (orders, accuracy and range: see there).
//
//   dw[n][i][j][d] = sum_v g[v][n] x[v + i W + j][d],   v = p W + q
// with g = 0 in the columns q >= Wo: a contraction over the pixels, whose two
// operands both have the pixel as their slow index.  They are staged in the chunk
// planes of the forward, [8 channels][pixel][16 bytes], and read as MN-major
// operands (core matrix: 8 pixels x 16 bytes; SBO = stride between 8-channel
// groups, LBO = 128 bytes between groups of 8 pixels):
//   B (N = 8 FWP): one plane of x, its groups the taps: SBO = 16 bytes, the same
//     plane started one pixel later, so no tap is ever copied;
//   A (M = 128): the planes of g's orders one under the other, so that one MMA
//     forms several of the six products:
//     NB = 64 filters: rows [g1 g2] with x1 -> D0, x2 -> D1, x3 -> D1, and [g3 0]
//                      with x1 -> D1
//     NB = 32:         rows [g1 g2 g3 0] with x1 -> D0, x2 -> D1, x3 -> D1
// D0 holds order 0 (and the row blocks of g2, g3 their own), D1 only smaller ones.
// The row blocks stay separate sums: each is a partial result of the reduction
// that adds the CTAs' sums up (fixed order, as before).
//
// An MMA of N = 64 takes 48 cycles (12 % of the tensor core's rate is lost to the
// reads of A), four of them do 64 x 56 x 16 multiply-adds for a 7-wide filter: 600
// FLOP per cycle and SM, where the FMA kernel reached 145.  256x256x16 * 64x7x7: 128 us
// with the FMA kernel, 67 us with this one (reduction and the FMA kernel's empty
// launch included); 512x512x32 * 256x5x5: 2148 and 1039.
//
// A CTA takes one filter row i, NCOMB planes of x, one tap group, one tile of NB
// filters and a run of chunks of KPX pixels.  A chunk is one accumulation chunk
// (KPX / 16 steps).  Warps 0..7 add the chunk sums up in FP32 registers, warps 8..13
// split g and x, one thread each of warps 14 and 15 issues the MMAs (of plane 0 and
// 1, or of D0 and D1): two threads never add to the same accumulator, so the order
// of the sums is fixed.
//
// A non-zero |v| < 2^-100, whose third part could fall below the BF16 range, or a
// non-finite sum sets the CTA's flag, and the FMA kernel launched next, which
// otherwise returns at once, computes the result.  x is split as 2^32 x and the sums
// multiplied by 2^-32 (both exact but for results below the normal range): without
// that, products near 2^-126 lost the small orders (error at 2^-130 2.4 times the FMA
// kernel's, now 0.13 times; 512x512x32 * 256x5x5 1027 to 1039 us, others unchanged).

#define FBC_F3_TINY ((27u << 24) - 1u)   // 2 * bits(2^-100) - 1
#define FBC_F3DW_UP 4294967296.f         // 2^32, of x: keeps products near 2^-126 in range

template <int FH_, int FW_, int C_, int NF_, int MASK_, int NB_, int NCOMB_, int JT_, int KPX_>
struct FbcF3DwCfg {
    static constexpr int FH = FH_, FW = FW_, C = C_, NF = NF_, MASK = MASK_, NB = NB_, NCOMB = NCOMB_, JT = JT_, KPX = KPX_;
    static constexpr int FWP = (JT + 1) / 2 * 2;             // taps of an operand (N = 8 FWP is a multiple of 16)
    static constexpr int NN = 8 * FWP;
    static constexpr int NTG = (FW + JT - 1) / JT;           // tap groups
    static constexpr int NCP = (C + 8 * NCOMB - 1) / (8 * NCOMB);   // plane groups
    static constexpr int NTN = (NF + NB - 1) / NB;           // filter tiles
    static constexpr int NH = NB == 64 ? 2 : 3;              // row blocks that hold sums
    static constexpr int STEPS = KPX / 16;
    static constexpr unsigned GPLANE = KPX * 16 + 16;        // padded by one chunk: banks
    static constexpr int GDATA = 3 * NB / 8;                 // planes with data, then zero planes
    static constexpr int GPLANES = NB == 64 ? 32 : 16;
    static constexpr int LS = KPX + FWP - 1;                 // slab pixels of x
    static constexpr int LP = NCOMB == 2 ? (LS + 3) / 8 * 8 + 4 : LS;
    static constexpr unsigned XPLANE = LP * 16;
    static constexpr unsigned XORD = NCOMB * XPLANE;
    static constexpr unsigned GBYTES = GPLANES * GPLANE;
    static constexpr unsigned SLOT = (GBYTES + 3 * XORD + 127) / 128 * 128;
    static constexpr int NS = 227 * 1024 - 2048 >= 4 * SLOT ? 4 : 227 * 1024 - 2048 >= 3 * SLOT ? 3 : 2;
    static constexpr int NCT = 32 * FBC_F3DW_CONV_WARPS;
    static constexpr int QG = NB / 4, QX = 2 * NCOMB;        // quads per pixel
    static constexpr int KG = (KPX * QG + NCT - 1) / NCT, KX = (LS * QX + NCT - 1) / NCT;
    static constexpr int BUF = NCOMB * 2 * NN;               // TMEM columns of one accumulator set
    static constexpr unsigned TMEM = 2 * BUF <= 64 ? 64 : 2 * BUF <= 128 ? 128 : 2 * BUF <= 256 ? 256 : 512;
    static constexpr int HC = NCOMB * NN / 2;                // columns per accumulating warp
};

template <class G>
__device__ __forceinline__ void fbc_f32dw_body(const FbcF3DwParams& P) {
    __shared__ int s_abort, s_flag;
    __shared__ fbc_u32 s_tmem;
    __shared__ __align__(8) fbc_u64 s_bar[2 * G::NS + 6];
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const fbc_u32 sbase = fbc_smem_addr(fbc_tc_smem);
    const fbc_u32 full0 = fbc_smem_addr(s_bar), empty0 = full0 + 8u * G::NS;
    const fbc_u32 acc_full0 = empty0 + 8u * G::NS, acc_empty0 = acc_full0 + 16u, drain_bar = acc_empty0 + 16u;
    // this CTA's part: filter row, tap group, planes of x, filter tile, run of chunks
    int b = blockIdx.x;
    const int s = b % P.splits;
    b /= P.splits;
    const int fi = b % G::FH;
    b /= G::FH;
    const int tg = b % G::NTG;
    b /= G::NTG;
    const int ch0 = (b % G::NCP) * 8 * G::NCOMB;
    const int n0 = (b / G::NCP) * G::NB;
    const int c0 = (int)((long long)P.nchunk * s / P.splits), c1 = (int)((long long)P.nchunk * (s + 1) / P.splits);
    if (threadIdx.x == 0) {
        for (int k = 0; k < G::NS; ++k) {
            fbc_mbar_init(full0 + 8u * k, FBC_F3DW_CONV_WARPS);
            fbc_mbar_init(empty0 + 8u * k, 2);           // both issuers' commits
        }
        for (int k = 0; k < 2; ++k) {
            fbc_mbar_init(acc_full0 + 8u * k, 2);
            fbc_mbar_init(acc_empty0 + 8u * k, FBC_F3_EPI_WARPS);
            fbc_mbar_init(drain_bar + 8u * k, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        s_flag = 0;
    }
    if (warp == 15) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(fbc_smem_addr(&s_tmem)),
                     "n"(G::TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // the zero rows of A
    for (int k = 0; k < G::NS; ++k)
        for (unsigned o = G::GDATA * G::GPLANE + threadIdx.x * 16; o < G::GBYTES; o += FBC_F3DW_THREADS * 16)
            fbc_st_shared_v4(sbase + k * G::SLOT + o, 0u, 0u, 0u, 0u);
    fbc_fence_proxy_async_smem();
    fbc_tc_fence_before();
    __syncthreads();
    fbc_tc_fence_after();
    const fbc_u32 tmem = s_tmem;
    volatile int* abort_flag = &s_abort;
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp >= 8 && warp < 8 + FBC_F3DW_CONV_WARPS) {
        // ------------------------------------------------------------ converters
        const int ct = threadIdx.x - 8 * 32;
        float gb[G::KG][4], xb[G::KX][4], mb[G::MASK ? G::KG : 1][4];
        auto load = [&](int c) {
            const int v0 = c * G::KPX;
#pragma unroll
            for (int k = 0; k < G::KG; ++k) {
                const int it = ct + k * G::NCT;
                const int px = it / G::QG, n = n0 + it % G::QG * 4;
                const int v = v0 + px;
                const int p = P.W == 1 ? v : (int)(__umulhi((unsigned)v, P.w_mul) >> P.w_shift);
                const int q = v - p * P.W;
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                if (px < G::KPX && q < P.Wo && p < P.Ho && n < G::NF) {
                    const unsigned o = (unsigned)((p * P.Wo + q) * G::NF + n);
                    f = __ldg(reinterpret_cast<const float4*>(P.g + o));
                    if constexpr (G::MASK) {
                        const float4 t = __ldg(reinterpret_cast<const float4*>(P.m + o));
                        mb[k][0] = t.x; mb[k][1] = t.y; mb[k][2] = t.z; mb[k][3] = t.w;
                    }
                }
                gb[k][0] = f.x; gb[k][1] = f.y; gb[k][2] = f.z; gb[k][3] = f.w;
            }
#pragma unroll
            for (int k = 0; k < G::KX; ++k) {
                const int it = ct + k * G::NCT;
                const int px = it / G::QX, ch = ch0 + it % G::QX * 4;
                const int v = v0 + fi * P.W + tg * G::JT + px;
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                if (px < G::LS && v < P.H * P.W && ch < G::C)
                    f = __ldg(reinterpret_cast<const float4*>(P.x + (unsigned)(v * G::C + ch)));
                xb[k][0] = f.x; xb[k][1] = f.y; xb[k][2] = f.z; xb[k][3] = f.w;
            }
        };
        if (c0 < c1) load(c0);
        int sl = 0;
        fbc_u32 ph = 0, tiny = 0xFFFFFFFFu;   // the least of 2|v| - 1 as integers (zeros: the largest)
        auto look = [&](const float (&v)[4]) {
#pragma unroll
            for (int e = 0; e < 4; ++e) tiny = min(tiny, __float_as_uint(v[e]) * 2u - 1u);
        };
        for (int c = c0; c < c1; ++c) {
            if (!fbc_wait(empty0 + 8u * sl, ph ^ 1, P, abort_flag, FBC_F3_ERR_WAIT)) break;
            const fbc_u32 gd = sbase + (fbc_u32)sl * G::SLOT, xd = gd + G::GBYTES;
#pragma unroll
            for (int k = 0; k < G::KG; ++k) {
                const int it = ct + k * G::NCT;
                const int px = it / G::QG, q = it % G::QG;
                if ((k + 1) * G::NCT <= G::KPX * G::QG || px < G::KPX) {
                    if constexpr (G::MASK) {
                        // not as they are loaded: a chunk's loads have the chunk before it to
                        // land (500x341x16 * 64x5x4, clamped: 284 to 101 us; FMA kernel 227)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (!(mb[k][e] > P.lo && mb[k][e] < P.hi)) gb[k][e] = 0.f;
                    }
                    look(gb[k]);
                    fbc_f3_put(gb[k], gd + (fbc_u32)(q >> 1) * G::GPLANE + (fbc_u32)px * 16u + (fbc_u32)(q & 1) * 8u,
                               (G::NB / 8) * G::GPLANE);
                }
            }
#pragma unroll
            for (int k = 0; k < G::KX; ++k) {
                const int it = ct + k * G::NCT;
                const int px = it / G::QX, q = it % G::QX;
                if ((k + 1) * G::NCT <= G::LS * G::QX || px < G::LS) {
                    look(xb[k]);
                    fbc_f3_scale(xb[k], FBC_F3DW_UP);
                    fbc_f3_put(xb[k], xd + (fbc_u32)(q >> 1) * G::XPLANE + (fbc_u32)px * 16u + (fbc_u32)(q & 1) * 8u, G::XORD);
                }
            }
            fbc_fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && !(FBC_F3_DROP && warp == 8 && c == c0)) fbc_mbar_arrive(full0 + 8u * sl);
            if (++sl == G::NS) { sl = 0; ph ^= 1; }
            if (c + 1 < c1) load(c + 1);
        }
        if (tiny < FBC_F3_TINY) s_flag = 1;
    } else if (warp >= 14) {
        if (lane == 0) {
            // -------------------------------------------------------- MMA issuers
            const int r = warp - 14;
            const fbc_u32 idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |   // both operands MN-major
                                  ((fbc_u32)(G::NN >> 3) << 17) | ((128u >> 4) << 24);
            const fbc_u64 ad0 = fbc_smem_desc(sbase, 128, G::GPLANE);
            const fbc_u64 xd0 = fbc_smem_desc(sbase + G::GBYTES + (G::NCOMB == 2 ? r * G::XPLANE : 0u), 128, 16);
            const fbc_u32 ahi = (fbc_u32)(ad0 >> 32), xhi = (fbc_u32)(xd0 >> 32);
            int sl = 0, acc = 0;
            fbc_u32 ph = 0, accph = 0;
            bool ok = true, issued = false;
            for (int c = c0; c < c1; ++c) {
                if (!(ok = fbc_wait(acc_empty0 + 8u * acc, accph ^ 1, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                if (!(ok = fbc_wait(full0 + 8u * sl, ph, P, abort_flag, FBC_F3_ERR_WAIT))) break;
                fbc_tc_fence_after();
                issued = true;
                const fbc_u32 d0 = tmem + (fbc_u32)(acc * G::BUF + (G::NCOMB == 2 ? r * 2 * G::NN : 0)), d1 = d0 + G::NN;
                const fbc_u32 alo = (fbc_u32)ad0 + ((fbc_u32)sl * G::SLOT >> 4), xlo = (fbc_u32)xd0 + ((fbc_u32)sl * G::SLOT >> 4);
#pragma unroll
                for (int e = 0; e < G::STEPS; ++e) {
                    const fbc_u32 a = alo + e * 16, x1 = xlo + e * 16, x2 = x1 + (G::XORD >> 4), x3 = x2 + (G::XORD >> 4);
                    if (G::NCOMB == 2 || r == 0) fbc_umma_lo(d0, a, ahi, x1, xhi, idesc, e > 0 ? 1u : 0u);
                    if (G::NCOMB == 2 || r == 1) {
                        fbc_umma_lo(d1, a, ahi, x3, xhi, idesc, e > 0 ? 1u : 0u);
                        if constexpr (G::NB == 64) fbc_umma_lo(d1, a + (16 * G::GPLANE >> 4), ahi, x1, xhi, idesc, 1u);
                        fbc_umma_lo(d1, a, ahi, x2, xhi, idesc, 1u);
                    }
                }
                fbc_umma_commit<1>(empty0 + 8u * sl);
                fbc_umma_commit<1>(acc_full0 + 8u * acc);
                if (++sl == G::NS) { sl = 0; ph ^= 1; }
                acc ^= 1;
                if (acc == 0) accph ^= 1;
            }
            if (!ok && issued) {
                fbc_umma_commit<1>(drain_bar + 8u * r);
                fbc_wait_drain(drain_bar + 8u * r, 0, P);
            }
        }
    } else {
        // ------------------------------------------------------------ accumulate
        const int lq = warp & 3, half = warp >> 2;
        // NCOMB = 2: plane `half`; NCOMB = 1: half of the columns
        const fbc_u32 col = G::NCOMB == 2 ? half * 2 * G::NN : half * G::HC;
        const fbc_u32 trow = tmem + ((fbc_u32)(lq * 32) << 16) + col;
        float sum[G::HC];
#pragma unroll
        for (int k = 0; k < G::HC; ++k) sum[k] = 0.f;
        int acc = 0;
        fbc_u32 accph = 0;
        bool ok = true;
        for (int c = c0; c < c1; ++c) {
            if (!(ok = fbc_wait(acc_full0 + 8u * acc, accph, P, abort_flag, FBC_F3_ERR_WAIT))) break;
            fbc_tc_fence_after();
            const fbc_u32 ta = trow + (fbc_u32)(acc * G::BUF);
#pragma unroll
            for (int k = 0; k < G::HC; k += 8) {
                fbc_u32 r0[8], r1[8];
                fbc_tmem_ld32x32b_x8_async(ta + k, r0);
                fbc_tmem_ld32x32b_x8_async(ta + G::NN + k, r1);
                fbc_tmem_ld_wait();
                fbc_reg_fence8(r0);
                fbc_reg_fence8(r1);
#pragma unroll
                for (int e = 0; e < 8; ++e) sum[k + e] += __uint_as_float(r0[e]) + __uint_as_float(r1[e]);
            }
            fbc_tc_fence_before();
            __syncwarp();
            if (lane == 0) fbc_mbar_arrive(acc_empty0 + 8u * acc);
            acc ^= 1;
            if (acc == 0) accph ^= 1;
        }
        // row block h and filter n of this lane's accumulator row
        const int row = lq * 32 + lane;
        const int h = row / G::NB, n = n0 + row % G::NB;
        float z = 0.f;
#pragma unroll
        for (int k = 0; k < G::HC; ++k) z += sum[k] - sum[k];
        if (!(z == 0.f) || !ok) s_flag = 1;
#pragma unroll
        for (int k = 0; k < G::HC; ++k) sum[k] *= FBC_F3_DOWN;
        if (h < G::NH && n < G::NF) {
            float* dst = P.part + ((((long long)s * G::NH + h) * G::NF + n) * G::FH + fi) * (G::FW * G::C);
            const int ch = ch0 + (G::NCOMB == 2 ? half * 8 : 0);
#pragma unroll
            for (int k = 0; k < G::HC; k += 8) {
                const int j = (G::NCOMB == 2 ? 0 : half * (G::HC / 8)) + k / 8, tap = tg * G::JT + j;
                if (j >= G::JT || tap >= G::FW) continue;
#pragma unroll
                for (int e = 0; e < 8; e += 4)
                    if (ch + e < G::C)
                        *reinterpret_cast<float4*>(dst + tap * G::C + ch + e) =
                            make_float4(sum[k + e], sum[k + e + 1], sum[k + e + 2], sum[k + e + 3]);
            }
        }
    }
    __syncwarp();
    fbc_tc_fence_before();
    __syncthreads();
    fbc_tc_fence_after();
    if (threadIdx.x == 0) P.flags[blockIdx.x] = s_flag;
    if (warp == 15)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(G::TMEM));
}

// f32dw_params.h -- the launch parameters of the FP32 tensor-core dL/dw kernel,
// shared verbatim by the host (f32dw_kernel.cu) and by the NVRTC source
// (rtcg_f32dw.cuh).  Plain types only, no includes.
#ifndef FBC_F32DW_PARAMS_H
#define FBC_F32DW_PARAMS_H

#define FBC_F3DW_CONV_WARPS 6   // warps that split g and x
#define FBC_F3DW_THREADS 512    // with 8 accumulating warps and two MMA warps

struct FbcF3DwParams {
    const float* x;             // [H][W][C]
    const float* g;             // [Ho][Wo][NF]
    const float* m;             // clamp-mask source, shaped as g (MASK only)
    float* part;                // [splits][NH][NF][FH][FW][C] partial sums
    int* flags;                 // per CTA: 1 when a value was outside the split's range
    int* err;                   // host-mapped error word
    unsigned long long wait_ns; // bound of every mbarrier wait
    float lo, hi;
    int H, W, Ho, Wo;
    unsigned int w_mul;         // v / W == umulhi(v, w_mul) >> w_shift for 0 <= v < 2^31 (W > 1)
    int w_shift;
    int nchunk;                 // chunks of KPX virtual pixels p * W + q
    int splits;                 // CTAs that share them
};

#endif

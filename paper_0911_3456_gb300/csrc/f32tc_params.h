// f32tc_params.h -- the launch parameters of the FP32 tensor-core correlation
// kernel, shared verbatim by the host (f32tc_kernel.cu) and by the NVRTC source
// (rtcg_f32tc.cuh), which gets this text prepended.  Plain types only, no
// includes: NVRTC compiles it without system headers.
#ifndef FBC_F32TC_PARAMS_H
#define FBC_F32TC_PARAMS_H

#define FBC_F3_EPI_WARPS 8      // accumulating and storing warps (two per TMEM lane quarter)
#define FBC_F3_CONV_WARPS 5     // warps that split x
#define FBC_F3_THREADS 512      // and a bank producer and two MMA warps: 128 registers per thread
#define FBC_F3_BANK_THREADS 256 // threads per block of the bank split, one chunk each

struct FbcF3Params {
    const float* x;             // [in_h][in_w][C]
    const float* m;             // clamp-mask source, shaped as x (MASK only)
    const float* w;             // the bank [N][FH][FW][D] (FLIP reads it flipped and transposed)
    float* y;                   // [out_h][out_w][NF]
    unsigned char* bank;        // the split bank: [filter tile][unit][BSTAGE bytes]
    int* err;                   // host-mapped error word
    unsigned long long wait_ns; // bound of every mbarrier wait
    float lo, hi;
    int in_h, in_w, out_h, out_w;
    int pad_y, pad_x;           // zero border of x (dL/dx)
    int vw;                     // virtual row width of the pixel tiles: out_w + FW - 1
    unsigned int vw_mul;        // v / vw == umulhi(v, vw_mul) >> vw_shift for 0 <= v < 2^31 (vw > 1)
    int vw_shift;
    int mtiles;                 // 128-pixel tiles over ceil(out_h / R) * vw virtual pixels
    int nitems;                 // mtiles x filter tiles
    int na, nb;                 // A slots, B stages per issuer
    unsigned int b_off, bar_off;    // B ring and barrier table in shared memory (A ring at 0)
};

#endif

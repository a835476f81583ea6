// Declarations of the per-tile quantizer and the value conversions it shares with the attention pre-pass.
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"

namespace hyq {

constexpr int QUANT_MAX_JOBS = 96;           // Q, K and V of a ragged launch's sequences
constexpr int QUANT_FEW_JOBS = 3;            // (the list travels as a kernel parameter: a short one where that is enough)

// one tensor [heads][L][D]
struct QuantJob {
    const uint4* x;
    uint8_t* codes;
    float* scales;
    uint4 *v16, *vh16;                       // optional: V and V^ as fp16 [heads][L][D]
    uint8_t* wide;                           // optional (INT4): codes as e4m3 bytes [heads][L][D]
    int L, heads, format;
    int tile0;                               // first tile of the tensor in the launch
};
template <int MAX> struct QuantList {
    int n;
    QuantJob job[MAX];
};
typedef QuantList<QUANT_MAX_JOBS> QuantJobs;
int launch_quantize_jobs(const QuantJobs& jobs, int block_tokens, cudaStream_t st);

// two floats -> fp16 pair, saturated to the largest finite fp16: a value row beyond the documented range
// (|V| < 65504) then degrades the result instead of putting an infinity, and with it NaNs, into the output
__device__ __forceinline__ uint32_t f16x2_sat(float a, float b) {
    const __half2 h2 = __floats2half2_rn(fminf(fmaxf(a, -65504.0f), 65504.0f), fminf(fmaxf(b, -65504.0f), 65504.0f));
    return *reinterpret_cast<const uint32_t*>(&h2);
}

// four two's-complement nibbles -> four e4m3 bytes (-8 .. 7 are exact): byte permutes look the magnitudes of the
// non-negative and of the negative codes up by the low three bits, a third spreads the sign bits (32 x 32768 rows of Q and 8 x 32768 of K: the
// look-up by shifts took 102 us in launches of its own, the whole pre-pass now 88 us, 149 before)
__device__ __forceinline__ uint32_t nibbles_to_e4m3(uint32_t w) {
    const uint32_t sel = w & 0x7777u;
    const uint32_t pos = __byte_perm(0x44403800u, 0x4E4C4A48u, sel), neg = __byte_perm(0x4A4C4E50u, 0x38404448u, sel);
    uint32_t m;                                               // selector bit 3: the byte's sign, spread over the byte
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(m) : "r"(0x80u), "r"(w & 0x8888u));
    m &= 0x7F7F7F7Fu;                                         // 0x7F where the code is negative
    return ((pos & ~m) | (neg & m)) | ((m << 1) & 0x80808080u);
}

}  // namespace hyq

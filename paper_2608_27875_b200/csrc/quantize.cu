// Per-tile symmetric quantization (Algorithm 2, Stage 2).
//
// One CTA of 2 * BT threads owns one tile of BT (32, 64 or 128) tokens x 128 channels: contiguous bf16
// (16 KB for the default 64 tokens).  Each thread keeps its 64 elements in registers (4 groups of 16
// consecutive channels, 32-byte loads), the tile absmax is a warp-shuffle reduction plus one
// shared-memory step across the 4 warps, and the codes leave as 16-byte (8-bit formats) or
// 8-byte (INT4) vector stores.  The tile is read once and written once: HBM-bound.
//
// One launch covers any number of tensors (QuantJob: the Q, K and V of a call, of every prompt of a ragged batch), whose
// tiles are numbered through; a tile looks its tensor up.  Inside the whole-path call a job may also write what the
// attention kernel streams - V and V^ as fp16, INT4 codes widened to e4m3 bytes - while the tile is in registers.
//
// Arithmetic is fp32 with one IEEE rounding per operation (no FMA contraction, no fast-math):
//   scale = absmax / c ; inv = c / absmax ; code = rint(x * inv), which cannot leave [-c, c], or e4m3(x * inv).
#include "quantize.cuh"

namespace hyq {

constexpr int QUANT_GROUPS = 4;                       // groups of 16 elements per thread

template <int FMT, int BT, bool EXTRAS>
__device__ __forceinline__ void quantize_tile(const QuantJob& job, int tile) {     // tile: head * nb + n
    constexpr int QUANT_THREADS = 2 * BT;
    const int nb = (job.L + BT - 1) / BT;
    const long head = tile / nb;
    const int t0 = (tile - (int)head * nb) * BT;
    const int tokens = min(BT, job.L - t0);
    const int n_elems = tokens * HYQ_D;
    const long elem0 = (head * job.L + t0) * (long)HYQ_D;
    const uint4* src = job.x + elem0 / 8;

    uint4 r[QUANT_GROUPS][2];
    uint32_t mx = 0u;
#pragma unroll
    for (int gi = 0; gi < QUANT_GROUPS; ++gi) {
        const int e = (threadIdx.x + gi * QUANT_THREADS) * 16;
        if (e < n_elems) {
            r[gi][0] = __ldg(src + e / 8);
            r[gi][1] = __ldg(src + e / 8 + 1);
        } else {
            r[gi][0] = make_uint4(0, 0, 0, 0);
            r[gi][1] = make_uint4(0, 0, 0, 0);
        }
        const uint32_t* w = reinterpret_cast<const uint32_t*>(&r[gi][0]);
#pragma unroll
        for (int c = 0; c < 8; ++c) mx = amax_pair(mx, w[c]);
    }
    mx = amax_warp(mx);
    __shared__ uint32_t warp_max[QUANT_THREADS / 32];
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < QUANT_THREADS / 32; ++w) mx = max(mx, warp_max[w]);
    const float amax = __uint_as_float(mx << 16);

    constexpr float c = (FMT == HYQ_FMT_INT8) ? 127.0f : (FMT == HYQ_FMT_FP8_E4M3) ? 448.0f : 7.0f;
    const bool dead = !(amax >= 0x1p-100f);
    const float inv = dead ? 0.0f : __fdiv_rn(c, amax), scale = dead ? 0.0f : __fdiv_rn(amax, c);
    if (threadIdx.x == 0) {
        job.scales[tile] = scale;
        if (EXTRAS && job.kv_fac) {
            float* fac = reinterpret_cast<float*>(job.kv_fac + tile);
            if (FMT != HYQ_FMT_INT4 && job.vh16) {
                const float2 rest = value_rest(scale);
                fac[1] = rest.x; fac[2] = rest.y;
            } else {
                fac[0] = scale;
            }
        }
    }
    const float vf = value_factor(scale);

    constexpr int ROW_BYTES = (FMT == HYQ_FMT_INT4) ? HYQ_D / 2 : HYQ_D;
    uint8_t* dst = job.codes + (head * job.L + t0) * (long)ROW_BYTES;
#pragma unroll
    for (int gi = 0; gi < QUANT_GROUPS; ++gi) {
        const int e = (threadIdx.x + gi * QUANT_THREADS) * 16;
        if (e >= n_elems) continue;
        const uint32_t* w = reinterpret_cast<const uint32_t*>(&r[gi][0]);
        uint32_t vh[8];                                  // V^ as fp16 pairs
        if (FMT == HYQ_FMT_FP8_E4M3) {
            const uint4 o = quant16_e4m3(w, inv, dead);
            *reinterpret_cast<uint4*>(dst + e) = o;
            if (EXTRAS && job.vh16) {
                const uint32_t oc[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int c2 = 0; c2 < 8; ++c2) {
                    const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)((oc[c2 >> 1] >> (16 * (c2 & 1))) & 0xFFFFu), __NV_E4M3);
                    const float2 ff = __half22float2(__half2(hr));
                    vh[c2] = f16x2_sat(ff.x * vf, ff.y * vf);
                }
            }
        } else if (FMT == HYQ_FMT_INT8) {
            *reinterpret_cast<uint4*>(dst + e) = quant16_int8(w, inv);
            if (EXTRAS && job.vh16) {
#pragma unroll
                for (int c2 = 0; c2 < 8; ++c2) {
                    const uint2 q = round_pair(w[c2], inv);
                    vh[c2] = f16x2_sat(rounded_value(q.x) * vf, rounded_value(q.y) * vf);
                }
            }
        } else {
            const uint2 o = quant16_int4(w, inv);
            *reinterpret_cast<uint2*>(dst + e / 2) = o;
            if (EXTRAS && job.wide)
                *reinterpret_cast<uint4*>(job.wide + elem0 + e) = make_uint4(nibbles_to_e4m3(o.x), nibbles_to_e4m3(o.x >> 16),
                                                                             nibbles_to_e4m3(o.y), nibbles_to_e4m3(o.y >> 16));
        }
        if (EXTRAS && FMT != HYQ_FMT_INT4 && job.vh16) {
            uint4* dh = job.vh16 + (elem0 + e) / 8;
            dh[0] = make_uint4(vh[0], vh[1], vh[2], vh[3]);
            dh[1] = make_uint4(vh[4], vh[5], vh[6], vh[7]);
            uint4* dv = job.v16 + (elem0 + e) / 8;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const uint32_t* x = w + 4 * half;
                dv[half] = make_uint4(f16x2_sat(bf16_lo(x[0]), bf16_hi(x[0])), f16x2_sat(bf16_lo(x[1]), bf16_hi(x[1])),
                                      f16x2_sat(bf16_lo(x[2]), bf16_hi(x[2])), f16x2_sat(bf16_lo(x[3]), bf16_hi(x[3])));
            }
        }
    }
}

// (format and extras are compile-time: with all of them in one kernel the registers of the largest cost every tile a
// fifth; a call with two formats takes two launches)
template <int FMT, int BT, bool EXTRAS, int MAX>
__global__ void __launch_bounds__(2 * BT)
quantize_kernel(const __grid_constant__ QuantList<MAX> jobs) {
    if (jobs.beside) pdl_launch_dependents();             // (a second launch, for the other format)
    else pdl_wait();
    int lo = 0, hi = jobs.n - 1;                          // the job whose tiles this one is among
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs.job[mid].tile0 <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    quantize_tile<FMT, BT, EXTRAS>(jobs.job[lo], blockIdx.x - jobs.job[lo].tile0);
    // one block's wait is enough: the kernel behind this one waits for all its blocks, and so for the kernels before it
    if (jobs.beside && blockIdx.x == 0) pdl_wait();
}

template <int FMT, int BT, bool EXTRAS>
static int launch_quantize_bt(const QuantJobs& jobs, long tiles, cudaStream_t st) {
    if (jobs.n > QUANT_FEW_JOBS)
        return launch_pdl(quantize_kernel<FMT, BT, EXTRAS, QUANT_MAX_JOBS>, dim3((unsigned)tiles), dim3(2 * BT), 0, st, jobs);
    QuantList<QUANT_FEW_JOBS> few;
    few.n = jobs.n; few.beside = jobs.beside;
    for (int j = 0; j < jobs.n; ++j) few.job[j] = jobs.job[j];
    return launch_pdl(quantize_kernel<FMT, BT, EXTRAS, QUANT_FEW_JOBS>, dim3((unsigned)tiles), dim3(2 * BT), 0, st, few);
}

// the jobs of one format
template <int FMT>
static int launch_quantize_fmt(const QuantJobs& all, int block_tokens, cudaStream_t st) {
    QuantJobs jobs;
    jobs.n = 0; jobs.beside = all.beside;
    long tiles = 0;
    bool extras = false;
    for (int j = 0; j < all.n; ++j) {
        if (all.job[j].format != FMT) continue;
        QuantJob& q = jobs.job[jobs.n++] = all.job[j];
        q.tile0 = (int)tiles;
        tiles += (long)q.heads * ((q.L + block_tokens - 1) / block_tokens);
        if (tiles > 0x7fffffffL) return HYQ_ERR_INVALID_ARG;
        extras |= q.vh16 != nullptr || q.wide != nullptr || q.kv_fac != nullptr;
    }
    if (tiles == 0) return HYQ_OK;
#define HYQ_QUANT(BT_) (extras ? launch_quantize_bt<FMT, BT_, true>(jobs, tiles, st) : launch_quantize_bt<FMT, BT_, false>(jobs, tiles, st))
    return block_tokens == 32 ? HYQ_QUANT(32) : block_tokens == 64 ? HYQ_QUANT(64) : block_tokens == 128 ? HYQ_QUANT(128) : HYQ_ERR_UNSUPPORTED;
#undef HYQ_QUANT
}

int launch_quantize_jobs(const QuantJobs& jobs, int block_tokens, cudaStream_t st) {
    int rc = launch_quantize_fmt<HYQ_FMT_INT8>(jobs, block_tokens, st);
    if (rc == HYQ_OK) rc = launch_quantize_fmt<HYQ_FMT_INT4>(jobs, block_tokens, st);
    if (rc == HYQ_OK) rc = launch_quantize_fmt<HYQ_FMT_FP8_E4M3>(jobs, block_tokens, st);
    return rc;
}

int launch_quantize(const void* x, long n_heads, int L, int block_tokens, int format, void* codes, float* scales, cudaStream_t st) {
    if (n_heads > 0x7fffffffL) return HYQ_ERR_INVALID_ARG;
    QuantJobs jobs;
    jobs.n = 1; jobs.beside = 0;
    QuantJob& j = jobs.job[0] = QuantJob{};
    j.x = static_cast<const uint4*>(x); j.codes = static_cast<uint8_t*>(codes); j.scales = scales;
    j.L = L; j.heads = (int)n_heads; j.format = format;
    return launch_quantize_jobs(jobs, block_tokens, st);
}

}  // namespace hyq

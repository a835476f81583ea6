// Column-mass vertical-line selector (Eq. 4-5): S(p) = sum over a set of tail queries of their softmax
// probability on key p, then top-k over the non-window prefix.
//
// The scores decide an index set that has to match the reference bit for bit, so the arithmetic is fixed
// operation by operation, all fp64 with explicit round-to-nearest intrinsics (no contraction):
//   s       = (fma chain over channels 0..127 from 0) * alpha
//   exp     = exp_det: two-part reduction by ln 2, degree-13 Taylor polynomial by Horner fma, exact 2^n scaling
//   row sum = per chunk of 64 keys: m_c = max, z_c = pairwise tree over exp(s - m_c) (the xor butterfly of a warp
//             IS that tree, the two warps of a CTA are its last level); then m = max m_c and
//             Z = sum_c z_c * exp(m_c - m) in ascending chunk order
//   S(p)    = sum over the queries in ascending order of exp(s - m_t) / Z_t
// Three kernels: chunk statistics (one pass over Q.K^T), their combination per query row, column sums (a second
// pass over the prefix columns); then the radix top-k of the Algorithm-1 selector.  Work is n_queries * L * 128
// fp64 fma per head and pass - a pre-pass for a handful of tail queries, not a second attention.
//
// Both passes use the same tile: a CTA of two warps owns 128 consecutive keys (two chunks) of one query head; a warp
// owns a chunk, each thread two keys of it (32 apart) against MASS_TQ queries at a time.  Bound by the fp64 pipe (64 fma
// per clock and SM): 2 x 8 independent chains per thread, eight broadcast loads of q for 32 fma, operands
// that need no conversion (select_common.cuh).  One key per thread with converted operands had the broadcasts and the
// conversions beside them: 12007 keys, 32 heads, 16 queries 241 + 85 + 244 us for the three kernels, now 135 + 11 + 139.
#include "select_common.cuh"

namespace hyq {

constexpr int MASS_KEYS = 64;        // keys per chunk of the row-sum definition
constexpr int MASS_CHUNKS = 2;       // chunks (warps) per CTA
constexpr int MASS_THREADS = 32 * MASS_CHUNKS;
constexpr int MASS_CTA_KEYS = MASS_KEYS * MASS_CHUNKS;
constexpr int MASS_TQ = 8;           // queries scored together
constexpr int MASS_QTILE = 16;       // query rows staged in shared memory at a time
constexpr int MASS_PITCH = HYQ_D / 8 + 1;                                   // 16-byte pieces per staged key row (conflict-free)
constexpr int MASS_SMEM = MASS_CTA_KEYS * MASS_PITCH * 16 + MASS_QTILE * HYQ_D * 8;

__device__ __forceinline__ double exp_det(double x) {
    if (!(x >= -690.0)) return 0.0;
    const double n = rint(__dmul_rn(x, 1.4426950408889634));
    double r = __fma_rn(n, -6.93147180369123816490e-01, x);
    r = __fma_rn(n, -1.90821492927058770002e-10, r);
    double p = 1.0 / 6227020800.0;
    p = __fma_rn(p, r, 1.0 / 479001600.0);
    p = __fma_rn(p, r, 1.0 / 39916800.0);
    p = __fma_rn(p, r, 1.0 / 3628800.0);
    p = __fma_rn(p, r, 1.0 / 362880.0);
    p = __fma_rn(p, r, 1.0 / 40320.0);
    p = __fma_rn(p, r, 1.0 / 5040.0);
    p = __fma_rn(p, r, 1.0 / 720.0);
    p = __fma_rn(p, r, 1.0 / 120.0);
    p = __fma_rn(p, r, 1.0 / 24.0);
    p = __fma_rn(p, r, 1.0 / 6.0);
    p = __fma_rn(p, r, 0.5);
    p = __fma_rn(p, r, 1.0);
    p = __fma_rn(p, r, 1.0);
    return __dmul_rn(p, __longlong_as_double(((long long)n + 1023) << 52));
}

// keys [j0, j0 + 128) of a head -> shared memory; rows past `last` repeat it
__device__ __forceinline__ void stage_keys(const __nv_bfloat16* kh, int j0, int last, uint4* ktile) {
    for (int v = threadIdx.x; v < MASS_CTA_KEYS * (HYQ_D / 8); v += MASS_THREADS)
        ktile[(v >> 4) * MASS_PITCH + (v & 15)] = __ldg(reinterpret_cast<const uint4*>(kh + (long)min(j0 + (v >> 4), last) * HYQ_D) + (v & 15));
}

// n query rows (zeros up to a multiple of MASS_TQ) -> shared memory as doubles scaled by 2^896
__device__ __forceinline__ void stage_queries(const __nv_bfloat16* qrows, int n, double* qd) {
    const int n_pad = (n + MASS_TQ - 1) / MASS_TQ * MASS_TQ;
    for (int e = threadIdx.x; e < n_pad * HYQ_D; e += MASS_THREADS) qd[e] = e < n * HYQ_D ? (double)__bfloat162float(qrows[e]) * K_UNIT : 0.0;
}

// scores of this thread's two keys against MASS_TQ staged query rows: independent fma chains in channel order
__device__ __forceinline__ void score_queries(const uint4* krow, const double* qd, double alpha, double (&s)[2][MASS_TQ]) {
#pragma unroll
    for (int c = 0; c < MASS_TQ; ++c) s[0][c] = s[1][c] = 0.0;
#pragma unroll 1
    for (int v = 0; v < HYQ_D / 8; ++v) {
        const uint4 ka = krow[v], kb = krow[32 * MASS_PITCH + v];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const uint32_t xa = w == 0 ? ka.x : w == 1 ? ka.y : w == 2 ? ka.z : ka.w, xb = w == 0 ? kb.x : w == 1 ? kb.y : w == 2 ? kb.z : kb.w;
            const double a0 = bf16_small(xa << 16), a1 = bf16_small(xa & 0xFFFF0000u);
            const double b0 = bf16_small(xb << 16), b1 = bf16_small(xb & 0xFFFF0000u);
#pragma unroll
            for (int c = 0; c < MASS_TQ; ++c) {
                const double2 qv = *reinterpret_cast<const double2*>(qd + c * HYQ_D + 8 * v + 2 * w);
                s[0][c] = __fma_rn(qv.x, a0, s[0][c]);
                s[1][c] = __fma_rn(qv.x, b0, s[1][c]);
                s[0][c] = __fma_rn(qv.y, a1, s[0][c]);
                s[1][c] = __fma_rn(qv.y, b1, s[1][c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < MASS_TQ; ++c) { s[0][c] = __dmul_rn(s[0][c], alpha); s[1][c] = __dmul_rn(s[1][c], alpha); }
}

// Pass 1: per (query row, chunk) the chunk maximum and the tree sum of exp(s - max).
__global__ void __launch_bounds__(MASS_THREADS)
mass_chunk_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ kmat, int Hq, int Hkv, int Lq,
                  int Lk, int nT, int n_chunks, double alpha, double* __restrict__ chunk_m, double* __restrict__ chunk_z) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint4* ktile = reinterpret_cast<uint4*>(smem_raw);
    double* qd = reinterpret_cast<double*>(smem_raw + MASS_CTA_KEYS * MASS_PITCH * 16);     // [MASS_QTILE][D]
    pdl_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per_head = (n_chunks + MASS_CHUNKS - 1) / MASS_CHUNKS, block = blockIdx.x % per_head;
    const long bh = blockIdx.x / per_head;                             // b * Hq + query head
    const int chunk = block * MASS_CHUNKS + wid, j = chunk * MASS_KEYS + lane;      // this thread's keys: j, j + 32
    stage_keys(kmat + bh / (Hq / Hkv) * Lk * HYQ_D, block * MASS_CTA_KEYS, Lk - 1, ktile);
    const uint4* krow = ktile + (wid * MASS_KEYS + lane) * MASS_PITCH;
    const int pos0 = Lk - nT;                                          // position of the first query of the set
    const __nv_bfloat16* qhead = q + (bh * Lq + (Lq - nT)) * HYQ_D;
    for (int t0 = 0; t0 < nT; t0 += MASS_QTILE) {
        const int nt = min(MASS_QTILE, nT - t0);
        __syncthreads();
        stage_queries(qhead + (long)t0 * HYQ_D, nt, qd);
        __syncthreads();
        for (int tq = 0; tq < nt; tq += MASS_TQ) {
            double s[2][MASS_TQ], m[MASS_TQ], z[2][MASS_TQ];
            score_queries(krow, qd + tq * HYQ_D, alpha, s);
#pragma unroll
            for (int c = 0; c < MASS_TQ; ++c) {
                const int pos = pos0 + t0 + tq + c;                    // causal: keys beyond it are not visible to this query
                if (j > pos) s[0][c] = -INFINITY;
                if (j + 32 > pos) s[1][c] = -INFINITY;
                m[c] = fmax(s[0][c], s[1][c]);
            }
            // maximum over the warp: every step halves the number of queries a lane looks after (lane's query: c_of(lane))
            // and the results are handed back to all lanes
#pragma unroll
            for (int o = 16, n = MASS_TQ; o > 0; o >>= 1) {
                if (n > 1) {
                    n >>= 1;
#pragma unroll
                    for (int c = 0; c < n; ++c) {
                        const bool up = (lane & o) != 0;
                        const double give = up ? m[c] : m[c + n], keep = up ? m[c + n] : m[c];
                        m[c] = fmax(keep, __shfl_xor_sync(0xffffffffu, give, o));
                    }
                } else {
                    m[0] = fmax(m[0], __shfl_xor_sync(0xffffffffu, m[0], o));
                }
            }
            // lane bits 4, 3, 2 chose halves of 8, 4, 2 queries: query c sits on the lanes with bits (4, 3, 2) = c
            const double m_own = m[0];
#pragma unroll
            for (int c = 0; c < MASS_TQ; ++c) {
                m[c] = __shfl_sync(0xffffffffu, m_own, c << 2);
                z[0][c] = s[0][c] == -INFINITY ? 0.0 : exp_det(__dsub_rn(s[0][c], m[c]));
                z[1][c] = s[1][c] == -INFINITY ? 0.0 : exp_det(__dsub_rn(s[1][c], m[c]));
            }
            // pairwise trees over the 32 keys of each half, neighbours first (sums of the same two numbers on either side, so
            // handing out the queries changes nothing); then the two halves
#pragma unroll
            for (int u = 0; u < 2; ++u) {
#pragma unroll
                for (int o = 1, n = MASS_TQ; o < 32; o <<= 1) {
                    if (n > 1) {
                        n >>= 1;
#pragma unroll
                        for (int c = 0; c < n; ++c) {
                            const bool up = (lane & o) != 0;
                            const double give = up ? z[u][c] : z[u][c + n], keep = up ? z[u][c + n] : z[u][c];
                            z[u][c] = __dadd_rn(keep, __shfl_xor_sync(0xffffffffu, give, o));
                        }
                    } else {
                        z[u][0] = __dadd_rn(z[u][0], __shfl_xor_sync(0xffffffffu, z[u][0], o));
                    }
                }
            }
            // query c sits on the lanes with bits (0, 1, 2) = c, most significant first
            const int c = (lane & 1) * 4 + (lane & 2) + ((lane >> 2) & 1);
            if (lane < 8 && tq + c < nt && chunk < n_chunks) {
                const long slot = (bh * nT + t0 + tq + c) * n_chunks + chunk;
                double mc = m[0];
#pragma unroll
                for (int e = 1; e < MASS_TQ; ++e) mc = c == e ? m[e] : mc;
                chunk_m[slot] = mc;
                chunk_z[slot] = __dadd_rn(z[0][0], z[1][0]);
            }
        }
    }
}

// Row maximum and row sum from the chunk statistics: one warp per (b, h, query); the terms of the sum in parallel, the
// additions in ascending chunk order.
__global__ void __launch_bounds__(128)
mass_combine_kernel(const double* __restrict__ chunk_m, const double* __restrict__ chunk_z, long rows,
                    int nT, int Lk, int n_chunks, double* __restrict__ row_mz) {
    pdl_wait();
    const long row = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;   // (bh * nT + t)
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    const int t = (int)(row % nT);
    const int nc = (Lk - nT + t) / MASS_KEYS + 1;                      // chunks that hold a visible key
    const double* cm = chunk_m + row * n_chunks;
    const double* cz = chunk_z + row * n_chunks;
    double m = -INFINITY;
    for (int c = lane; c < nc; c += 32) m = fmax(m, __ldg(cm + c));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    double Z = 0.0;
    for (int c0 = 0; c0 < nc; c0 += 32) {
        const int c = c0 + lane;
        const double term = c < nc ? __dmul_rn(__ldg(cz + c), exp_det(__dsub_rn(__ldg(cm + c), m))) : 0.0;
        const int n = min(32, nc - c0);
#pragma unroll 8
        for (int i = 0; i < n; ++i) Z = __dadd_rn(Z, __shfl_sync(0xffffffffu, term, i));
    }
    if (lane == 0) {
        row_mz[2 * row] = m;
        row_mz[2 * row + 1] = Z;
    }
}

// Pass 2: S(p) for the prefix keys, queries in ascending order.
__global__ void __launch_bounds__(MASS_THREADS)
mass_column_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ kmat, int Hq, int Hkv, int Lq,
                   int Lk, int P, int nT, double alpha, const double* __restrict__ row_mz, double* __restrict__ scores) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint4* ktile = reinterpret_cast<uint4*>(smem_raw);
    double* qd = reinterpret_cast<double*>(smem_raw + MASS_CTA_KEYS * MASS_PITCH * 16);     // [MASS_QTILE][D]
    pdl_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per_head = (P + MASS_CTA_KEYS - 1) / MASS_CTA_KEYS, block = blockIdx.x % per_head;
    const long bh = blockIdx.x / per_head;
    const int p = block * MASS_CTA_KEYS + wid * MASS_KEYS + lane;  // this thread's keys: p, p + 32
    stage_keys(kmat + bh / (Hq / Hkv) * Lk * HYQ_D, block * MASS_CTA_KEYS, P - 1, ktile);
    const uint4* krow = ktile + (wid * MASS_KEYS + lane) * MASS_PITCH;
    const __nv_bfloat16* qhead = q + (bh * Lq + (Lq - nT)) * HYQ_D;
    double S0 = 0.0, S1 = 0.0;
    for (int t0 = 0; t0 < nT; t0 += MASS_QTILE) {
        const int nt = min(MASS_QTILE, nT - t0);
        __syncthreads();
        stage_queries(qhead + (long)t0 * HYQ_D, nt, qd);
        __syncthreads();
        for (int tq = 0; tq < nt; tq += MASS_TQ) {
            double s[2][MASS_TQ];
            score_queries(krow, qd + tq * HYQ_D, alpha, s);
            const double2* mz = reinterpret_cast<const double2*>(row_mz) + bh * nT + t0 + tq;
#pragma unroll
            for (int c = 0; c < MASS_TQ; ++c) {
                if (tq + c < nt) {
                    const double2 r = __ldg(mz + c);
                    S0 = __dadd_rn(S0, __ddiv_rn(exp_det(__dsub_rn(s[0][c], r.x)), r.y));
                    S1 = __dadd_rn(S1, __ddiv_rn(exp_det(__dsub_rn(s[1][c], r.x)), r.y));
                }
            }
        }
    }
    if (p < P) scores[bh * P + p] = S0;
    if (p + 32 < P) scores[bh * P + p + 32] = S1;
}

size_t select_mass_workspace_bytes(int B, int Hq, int Lk, int window, int n_queries) {
    const long P = (Lk - window > 0) ? Lk - window : 0;
    const long rows = (long)B * Hq * n_queries, n_chunks = (Lk + MASS_KEYS - 1) / MASS_KEYS;
    return align_up((size_t)B * Hq * P * sizeof(double), 256) + 2 * align_up((size_t)rows * n_chunks * sizeof(double), 256) +
           align_up((size_t)rows * 2 * sizeof(double), 256);
}

int launch_select_mass(const void* q, const void* k, int B, int Hq, int Hkv, int Lq, int Lk, int window, int n_queries,
                       int k_sel, double alpha, int32_t* idx_out, void* ws, cudaStream_t st) {
    const int P = Lk - window, nT = n_queries;
    const long rows = (long)B * Hq * nT;
    const int n_chunks = (Lk + MASS_KEYS - 1) / MASS_KEYS;
    char* base = static_cast<char*>(ws);
    double* scores = reinterpret_cast<double*>(base);
    base += align_up((size_t)B * Hq * P * sizeof(double), 256);
    double* chunk_m = reinterpret_cast<double*>(base);
    base += align_up((size_t)rows * n_chunks * sizeof(double), 256);
    double* chunk_z = reinterpret_cast<double*>(base);
    base += align_up((size_t)rows * n_chunks * sizeof(double), 256);
    double* row_mz = reinterpret_cast<double*>(base);
    const auto* qb = static_cast<const __nv_bfloat16*>(q);
    const auto* kb = static_cast<const __nv_bfloat16*>(k);

    if (cudaFuncSetAttribute(mass_chunk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MASS_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(mass_column_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, MASS_SMEM) != cudaSuccess)
        return HYQ_ERR_CUDA;
    const long blocks1 = (long)((n_chunks + MASS_CHUNKS - 1) / MASS_CHUNKS) * B * Hq, blocks2 = (long)((P + MASS_CTA_KEYS - 1) / MASS_CTA_KEYS) * B * Hq;
    if (blocks1 > 0x7fffffffL) return HYQ_ERR_UNSUPPORTED;
    int rc = launch_pdl(mass_chunk_kernel, dim3((unsigned)blocks1), dim3(MASS_THREADS), MASS_SMEM, st, qb, kb, Hq,
                        Hkv, Lq, Lk, nT, n_chunks, alpha, chunk_m, chunk_z);
    if (rc != HYQ_OK) return rc;
    rc = launch_pdl(mass_combine_kernel, dim3((unsigned)((rows + 3) / 4)), dim3(128), 0, st, chunk_m, chunk_z, rows, nT, Lk, n_chunks, row_mz);
    if (rc != HYQ_OK) return rc;
    rc = launch_pdl(mass_column_kernel, dim3((unsigned)blocks2), dim3(MASS_THREADS), MASS_SMEM, st, qb, kb, Hq, Hkv,
                    Lq, Lk, P, nT, alpha, row_mz, scores);
    if (rc != HYQ_OK) return rc;
    SelTable tab{};
    tab.n_seq = 1; tab.heads = B * Hq; tab.g = Hq / Hkv;
    tab.seq[0].P = P; tab.seq[0].k_sel = k_sel;
    return launch_topk_table(tab, scores, idx_out, st);
}

}  // namespace hyq

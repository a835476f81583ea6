// Column-mass vertical-line selector (Eq. 4-5): S(p) = sum over a set of tail queries of their softmax
// probability on key p, then top-k over the non-window prefix.
//
// The scores decide an index set that has to match the reference bit for bit, so the arithmetic is fixed
// operation by operation, all fp64 with explicit round-to-nearest intrinsics (no contraction):
//   s       = (fma chain over channels 0..127 from 0) * alpha
//   exp     = exp_det: two-part reduction by ln 2, degree-13 Taylor polynomial by Horner fma, exact 2^n scaling
//   row sum = per chunk of 64 keys: m_c = max, z_c = pairwise tree over exp(s - m_c) (neighbours
//             first, the two halves of the chunk last); then m = max m_c and
//             Z = sum_c z_c * exp(m_c - m) in ascending chunk order
//   S(p)    = sum over the queries in ascending order of exp(s - m_t) / Z_t
// Three kernels: the scores with the chunk statistics, the statistics' combination per query row, column sums; then the radix
// top-k of the Algorithm-1 selector.  Work is n_queries * L * 128 fp64 fma per head - a pre-pass for a handful of tail queries,
// not a second attention.  The scores of the prefix are kept for the column sums, which are then exponentials and
// divisions only (a score costs 128 fma, 7 ps of the whole GPU, against 16 bytes written and read, 2.4 ps from memory); a call goes
// through its heads in groups whose scores fit in L2.
//
// The score kernel multiplies with the fp64 matrix instruction, whose results are those of the fma chain in ascending order of
// the contraction index, bit for bit (not promised by its manual: the tests hold keys that agree up to 50 binary orders below
// their scores against it).  It runs at 18.4 T fma/s, the plain instruction
// at 15.3, of which its kernels saw half beside their conversions of bf16 bits and shared-memory loads (and doubles staged in shared
// memory, 8 x 4 instead of 2 x 8 chains per thread or twice the warps did not change that): one conversion now serves 16 queries.
// A warp owns a chunk of 64 keys against up to 16 queries.  12007 keys, 32 heads, 16 queries: 124 + 8 + 125 us for the three kernels
// with the scores computed twice on the plain pipe, now 85 + 8 + 26 (4 queries: 69 + 8 + 62, now 48 + 8 + 8).
#include "select_common.cuh"

namespace hyq {

constexpr int MASS_KEYS = 64;        // keys per chunk of the row-sum definition
constexpr int MASS_CHUNKS = 2;       // chunks (warps) per CTA
constexpr int MASS_THREADS = 32 * MASS_CHUNKS;
constexpr int MASS_CTA_KEYS = MASS_KEYS * MASS_CHUNKS;
constexpr int MASS_SLAB = 64;        // channels staged at a time: eight CTAs per SM (all 128: four, and 111 us instead of 85)
constexpr int MASS_KPITCH = MASS_SLAB + 16;                                // bf16 numbers per staged key row, and ...
constexpr int MASS_QPITCH = MASS_SLAB + 2;                                 // ... doubles per staged query row: no bank conflicts
constexpr int mass_smem(int qt) { return MASS_CTA_KEYS * MASS_KPITCH * 2 + 8 * qt * MASS_QPITCH * 8; }
constexpr long MASS_GROUP_BYTES = 96L << 20;                               // kept scores of a group of heads (one head at least)

// D[16 keys x 8 queries] += A[16 x 16 channels] . B[16 x 8]: lane 4 g + t holds keys g, g + 8 and channels t + 4 i of A (a[2 i],
// a[2 i + 1]), query g and channels t + 4 i of B, and keys g, g + 8 and queries 2 t, 2 t + 1 of D
__device__ __forceinline__ void mma_f64(double (&c)[4], const double (&a)[8], const double (&b)[4]) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7,%8,%9,%10,%11}, {%12,%13,%14,%15}, {%0,%1,%2,%3};"
                 : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
                 : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(a[4]), "d"(a[5]), "d"(a[6]), "d"(a[7]), "d"(b[0]), "d"(b[1]), "d"(b[2]), "d"(b[3]));
}

// Without a branch, so that several chains run side by side, and rounding to a whole number by an addition, whose low word is that
// number: the conversion instructions and the chains one after the other cost 5 us of 136 at the size above.
// (Below -690, at -infinity and for -infinity minus itself the result is 0.)
__device__ __forceinline__ double exp_det(double x) {
    constexpr double MAGIC = 6755399441055744.0;                      // 1.5 * 2^52
    const bool live = x >= -690.0;
    x = live ? x : 0.0;
    const double t = __dadd_rn(__dmul_rn(x, 1.4426950408889634), MAGIC), n = __dsub_rn(t, MAGIC);
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
    return live ? __dmul_rn(p, __hiloint2double((__double2loint(t) + 1023) << 20, 0)) : 0.0;
}

// Pass 1: the scores of the prefix keys, and per (query row, chunk) the chunk maximum and the tree sum of exp(s - max).
// Grid: key blocks of the heads from bh0 on, tiles of 8 QT queries.  The 16 channels of a step are staged in the order t + 4 i, t
// major, so that a lane reads its four at once.
template <int QT>
__global__ void __launch_bounds__(MASS_THREADS)
mass_score_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ kmat, int bh0, int g, int Lq,
                  int Lk, int P, int nT, int n_chunks, double alpha, double* __restrict__ kept, double* __restrict__ chunk_m,
                  double* __restrict__ chunk_z) {
    constexpr int QTILE = 8 * QT, TQ = 2 * QT;                         // queries per tile, per thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __nv_bfloat16* kt = reinterpret_cast<__nv_bfloat16*>(smem_raw);                             // scaled by 2^-896 when converted
    double* qd = reinterpret_cast<double*>(smem_raw + MASS_CTA_KEYS * MASS_KPITCH * 2);         // scaled by 2^896
    pdl_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, kg = lane >> 2, qg = lane & 3;
    const int blocks = (n_chunks + MASS_CHUNKS - 1) / MASS_CHUNKS, block = blockIdx.x % blocks, h = blockIdx.x / blocks;
    const int t0 = blockIdx.y * QTILE, nt = min(QTILE, nT - t0);
    const long bh = bh0 + h;                                           // b * Hq + query head
    const uint4* kh = reinterpret_cast<const uint4*>(kmat + bh / g * Lk * HYQ_D);
    const __nv_bfloat16* qrows = q + (bh * Lq + (Lq - nT + t0)) * HYQ_D;
    double acc[4][QT][4];
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int n = 0; n < QT; ++n) acc[mt][n][0] = acc[mt][n][1] = acc[mt][n][2] = acc[mt][n][3] = 0.0;
    const __nv_bfloat16* krow = kt + (wid * MASS_KEYS + kg) * MASS_KPITCH + qg * 4;
    const double* qrow = qd + kg * MASS_QPITCH + qg * 4;
#pragma unroll 1
    for (int d0 = 0; d0 < HYQ_D; d0 += MASS_SLAB) {
        if (d0 > 0) __syncthreads();
        constexpr int KB = MASS_SLAB / 16;                             // 16-channel blocks per row
#pragma unroll 4
        for (int v = threadIdx.x; v < MASS_CTA_KEYS * KB; v += MASS_THREADS) {
            const int row = v / KB, blk = v % KB;                      // (rows past the last repeat it)
            const uint4* src = kh + (long)min(block * MASS_CTA_KEYS + row, Lk - 1) * (HYQ_D / 8) + d0 / 8 + blk * 2;
            const uint4 x = __ldg(src), y = __ldg(src + 1);
            uint4* dst = reinterpret_cast<uint4*>(kt + row * MASS_KPITCH + blk * 16);
            dst[0] = make_uint4(__byte_perm(x.x, x.z, 0x5410), __byte_perm(y.x, y.z, 0x5410), __byte_perm(x.x, x.z, 0x7632), __byte_perm(y.x, y.z, 0x7632));
            dst[1] = make_uint4(__byte_perm(x.y, x.w, 0x5410), __byte_perm(y.y, y.w, 0x5410), __byte_perm(x.y, x.w, 0x7632), __byte_perm(y.y, y.w, 0x7632));
        }
#pragma unroll 4
        for (int e = threadIdx.x; e < QTILE * MASS_SLAB; e += MASS_THREADS) {
            const int row = e / MASS_SLAB, d = e % MASS_SLAB;
            qd[row * MASS_QPITCH + (d & ~15) + (d & 3) * 4 + ((d >> 2) & 3)] =
                row < nt ? (double)__bfloat162float(qrows[row * HYQ_D + d0 + d]) * K_UNIT : 0.0;
        }
        __syncthreads();
#pragma unroll 1
        for (int k0 = 0; k0 < MASS_SLAB; k0 += 16) {
            double b[QT][4];
#pragma unroll
            for (int n = 0; n < QT; ++n) {
                const double2 lo = *reinterpret_cast<const double2*>(qrow + 8 * n * MASS_QPITCH + k0), hi = *reinterpret_cast<const double2*>(qrow + 8 * n * MASS_QPITCH + k0 + 2);
                b[n][0] = lo.x; b[n][1] = lo.y; b[n][2] = hi.x; b[n][3] = hi.y;
            }
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                double a[8];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const uint2 w = *reinterpret_cast<const uint2*>(krow + (16 * mt + 8 * r) * MASS_KPITCH + k0);
                    a[r] = bf16_small(w.x << 16);
                    a[2 + r] = bf16_small(w.x & 0xFFFF0000u);
                    a[4 + r] = bf16_small(w.y << 16);
                    a[6 + r] = bf16_small(w.y & 0xFFFF0000u);
                }
#pragma unroll
                for (int n = 0; n < QT; ++n) mma_f64(acc[mt][n], a, b[n]);
            }
        }
    }
    // this thread's keys: j + 8 u; its queries: 8 n + 2 qg + e for c = 2 n + e
    const int chunk = block * MASS_CHUNKS + wid, j = chunk * MASS_KEYS + kg;
    auto query_of = [&](int c) -> int { return 8 * (c >> 1) + 2 * qg + (c & 1); };
    const bool edge = chunk * MASS_KEYS + MASS_KEYS - 1 > Lk - nT + t0;           // keys that not every query of the tile sees
    double s[8][TQ], m[TQ];
#pragma unroll
    for (int c = 0; c < TQ; ++c) {
        const int t = query_of(c), pos = Lk - nT + t0 + t;             // causal: keys beyond pos are not visible to this query
        double* row = kept + ((long)h * nT + t0 + t) * P;
        m[c] = -INFINITY;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const double x = __dmul_rn(acc[u >> 1][c >> 1][2 * (u & 1) + (c & 1)], alpha);
            if (t < nt && j + 8 * u < P) row[j + 8 * u] = x;
            s[u][c] = edge && j + 8 * u > pos ? -INFINITY : x;
            m[c] = s[u][c] > m[c] ? s[u][c] : m[c];
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) { const double v = __shfl_xor_sync(0xffffffffu, m[c], o); m[c] = v > m[c] ? v : m[c]; }
    }
    // Pairwise tree over the keys of each half of the chunk, neighbours first: the lowest three key bits across the lanes, the
    // next two in the thread, then the two halves.  Across the lanes every step halves the number of (query, half) items a
    // lane looks after, as long as there are several (sums of the same two numbers on either side, so handing them out changes nothing).
    constexpr int NI = 2 * TQ, LB = TQ == 4 ? 3 : 2;
    double z[NI][4];
#pragma unroll
    for (int c = 0; c < TQ; ++c)
#pragma unroll
        for (int u = 0; u < 8; ++u) z[2 * c + (u >> 2)][u & 3] = exp_det(__dsub_rn(s[u][c], m[c]));
#pragma unroll
    for (int o = 1, n = NI; o < 8; o <<= 1) {
        const bool halve = n > 1;
        if (halve) n >>= 1;
#pragma unroll
        for (int i = 0; i < n; ++i)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool up = (kg & o) != 0;
                const double give = !halve ? z[i][u] : up ? z[i][u] : z[i + n][u], keep = !halve ? z[i][u] : up ? z[i + n][u] : z[i][u];
                z[i][u] = __dadd_rn(keep, __shfl_xor_sync(0xffffffffu, give, 4 * o));
            }
    }
    const double zh = __dadd_rn(__dadd_rn(z[0][0], z[0][1]), __dadd_rn(z[0][2], z[0][3]));
    const double zc = __dadd_rn(zh, __shfl_xor_sync(0xffffffffu, zh, 4 << (LB - 1)));
    // item 2 c + half sits on the lanes whose lowest LB bits of the key group, lowest first, spell it
    int c = 0;
#pragma unroll
    for (int b = 0; b < LB - 1; ++b) c = 2 * c + ((kg >> b) & 1);
    const int t = query_of(c);
    if ((kg >> (LB - 1)) == 0 && t < nt && chunk < n_chunks) {
        const long slot = ((long)h * nT + t0 + t) * n_chunks + chunk;
        double mc = m[0];
#pragma unroll
        for (int e = 1; e < TQ; ++e) mc = c == e ? m[e] : mc;
        chunk_m[slot] = mc;
        chunk_z[slot] = zc;
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

// Pass 2: S(p) for the prefix keys, queries in ascending order; a thread per key.  (blockIdx.y: head of the group)
constexpr int MASS_SUM_THREADS = 128;
constexpr int MASS_SUM_AHEAD = 4;                                      // terms worked out side by side
__global__ void __launch_bounds__(MASS_SUM_THREADS)
mass_sum_kernel(const double* __restrict__ kept, const double* __restrict__ row_mz, int P, int nT, double* __restrict__ scores) {
    pdl_wait();
    const int p = blockIdx.x * MASS_SUM_THREADS + threadIdx.x;
    if (p >= P) return;
    const double* col = kept + (long)blockIdx.y * nT * P + p;
    const double2* mz = reinterpret_cast<const double2*>(row_mz) + (long)blockIdx.y * nT;
    double S = 0.0;
    for (int t0 = 0; t0 < nT; t0 += MASS_SUM_AHEAD) {
        double term[MASS_SUM_AHEAD];
#pragma unroll
        for (int c = 0; c < MASS_SUM_AHEAD; ++c) {
            const int t = min(t0 + c, nT - 1);
            const double2 r = __ldg(mz + t);
            term[c] = __ddiv_rn(exp_det(__dsub_rn(__ldg(col + (long)t * P), r.x)), r.y);
        }
#pragma unroll
        for (int c = 0; c < MASS_SUM_AHEAD; ++c)
            if (t0 + c < nT) S = __dadd_rn(S, term[c]);
    }
    scores[(long)blockIdx.y * P + p] = S;
}

// heads of one round of launches, and the workspace that follows from it
struct MassPlan {
    int heads;                       // heads per group
    size_t scores, kept, stats, mz;  // bytes
    size_t total() const { return scores + kept + 2 * stats + mz; }
};
static MassPlan mass_plan(int B, int Hq, int Lk, int window, int n_queries) {
    const long P = (Lk - window > 0) ? Lk - window : 0, per_head = (long)n_queries * P * (long)sizeof(double);
    const long all = (long)B * Hq, n_chunks = (Lk + MASS_KEYS - 1) / MASS_KEYS;
    MassPlan m;
    long heads = per_head > 0 ? MASS_GROUP_BYTES / per_head : all;
    heads = heads < 1 ? 1 : heads > all ? all : heads;
    heads = heads > 65535 ? 65535 : heads;                             // (a grid dimension of pass 2)
    m.heads = (int)heads;
    m.scores = align_up((size_t)all * P * sizeof(double), 256);
    m.kept = align_up((size_t)(heads * per_head), 256);
    m.stats = align_up((size_t)(heads * n_queries * n_chunks) * sizeof(double), 256);
    m.mz = align_up((size_t)(heads * n_queries) * 2 * sizeof(double), 256);
    return m;
}
size_t select_mass_workspace_bytes(int B, int Hq, int Lk, int window, int n_queries) { return mass_plan(B, Hq, Lk, window, n_queries).total(); }
// The query's answer: never less than that of a call with fewer heads, keys or queries.  (A group's heads are a whole number, so
// that a longer call may need less than a shorter one; here the groups are full and the statistics those of all heads.)
size_t select_mass_query_bytes(int B, int Hq, int Lk, int window, int n_queries) {
    const size_t P = Lk > window ? Lk - window : 0, all = (size_t)B * Hq, per_head = (size_t)n_queries * P * sizeof(double);
    const size_t n_chunks = (Lk + MASS_KEYS - 1) / MASS_KEYS, group = per_head > (size_t)MASS_GROUP_BYTES ? per_head : (size_t)MASS_GROUP_BYTES;
    return align_up(all * P * sizeof(double), 256) + align_up(all * per_head < group ? all * per_head : group, 256) +
           2 * align_up(all * n_queries * n_chunks * sizeof(double), 256) + align_up(all * n_queries * 2 * sizeof(double), 256);
}

int launch_select_mass(const void* q, const void* k, int B, int Hq, int Hkv, int Lq, int Lk, int window, int n_queries,
                       int k_sel, double alpha, int32_t* idx_out, void* ws, cudaStream_t st) {
    const int P = Lk - window, nT = n_queries, n_chunks = (Lk + MASS_KEYS - 1) / MASS_KEYS, g = Hq / Hkv;
    const MassPlan plan = mass_plan(B, Hq, Lk, window, nT);
    char* base = static_cast<char*>(ws);
    double* scores = reinterpret_cast<double*>(base);
    double* kept = reinterpret_cast<double*>(base += plan.scores);
    double* chunk_m = reinterpret_cast<double*>(base += plan.kept);
    double* chunk_z = reinterpret_cast<double*>(base += plan.stats);
    double* row_mz = reinterpret_cast<double*>(base += plan.stats);
    const auto* qb = static_cast<const __nv_bfloat16*>(q);
    const auto* kb = static_cast<const __nv_bfloat16*>(k);
    const int qt = nT > 8 ? 2 : 1, smem = mass_smem(qt);
    auto kern = qt == 2 ? mass_score_kernel<2> : mass_score_kernel<1>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return HYQ_ERR_CUDA;
    const long key_blocks = (n_chunks + MASS_CHUNKS - 1) / MASS_CHUNKS, q_tiles = (nT + 8 * qt - 1) / (8 * qt);
    if (key_blocks * plan.heads > 0x7fffffffL || q_tiles > 65535) return HYQ_ERR_UNSUPPORTED;
    for (int bh0 = 0; bh0 < B * Hq; bh0 += plan.heads) {
        const int heads = B * Hq - bh0 < plan.heads ? B * Hq - bh0 : plan.heads;
        const long rows = (long)heads * nT;
        int rc = launch_pdl(kern, dim3((unsigned)(key_blocks * heads), (unsigned)q_tiles), dim3(MASS_THREADS), smem, st, qb, kb, bh0, g, Lq, Lk, P,
                            nT, n_chunks, alpha, kept, chunk_m, chunk_z);
        if (rc != HYQ_OK) return rc;
        rc = launch_pdl(mass_combine_kernel, dim3((unsigned)((rows + 3) / 4)), dim3(128), 0, st, chunk_m, chunk_z, rows, nT, Lk, n_chunks, row_mz);
        if (rc != HYQ_OK) return rc;
        rc = launch_pdl(mass_sum_kernel, dim3((unsigned)((P + MASS_SUM_THREADS - 1) / MASS_SUM_THREADS), (unsigned)heads), dim3(MASS_SUM_THREADS), 0, st,
                        kept, row_mz, P, nT, scores + (long)bh0 * P);
        if (rc != HYQ_OK) return rc;
    }
    SelTable tab{};
    tab.n_seq = 1; tab.heads = B * Hq; tab.g = Hq / Hkv;
    tab.seq[0].P = P; tab.seq[0].k_sel = k_sel;
    return launch_topk_table(tab, scores, idx_out, st);
}

}  // namespace hyq

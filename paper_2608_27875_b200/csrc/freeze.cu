// Freeze (Algorithm 4): builds the hybrid KV cache of the decode stage from the prefill cache.
//
// One kernel, HBM-bound and read-once / write-once; a block either
//   - quantizes one group of G (32, 64 or 128) COMPACTED rows of one (b, kv head), K and V: finds the source rows (the
//     complement of the ascending vertical set) once for both, quantizes the two G x 128 groups with the arithmetic of
//     the per-tile quantizer, and writes K row-major and V in the fragment-major tile layout the decode kernel
//     loads straight into matrix-instruction operand registers; or
//   - copies vertical rows (by index) and window rows (a slice) as bf16.
// What kept it from the memory's rate was the chain search -> row numbers -> loads of 16 KB per CTA, and one conversion
// instruction per element.  One chain now serves 32 KB, all loads are issued before the first maximum, and rounding is an
// addition: 8 x 8 heads x 32768 rows (1.38 GB moved), INT4: 295 -> 242 us.
#include <string.h>

#include "decode_common.cuh"
#include "quantize.cuh"

namespace hyq {

constexpr int FRZ_THREADS = 128;     // append kernel; the quantizer runs 2 * G threads (64 elements of K and of V per thread)
constexpr int FRZ_QTHREADS_PER_SM = 768;    // quantizer threads resident per SM the register budget is set for (512: 285 us, 640: 272, 896: 262)

// Source position of compacted row p: p + j with j the number of vertical indices below it,
// i.e. the smallest j with idx[j] - j > p (idx ascending, so idx[j] - j never decreases).
__device__ __forceinline__ int source_row(const int32_t* __restrict__ idx, int k, int p) {
    int lo = 0, hi = k;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(idx + mid) - mid > p) hi = mid; else lo = mid + 1;
    }
    return p + lo;
}

struct FreezeParams {
    const uint4 *k, *v;
    const int32_t* idx;
    int N, W, k_vl, nQ, n_groups;
    long nQp, sK, sW;
    uint8_t *kq, *vq;
    float *ks, *vs;
    uint4 *k_vl_out, *v_vl_out, *k_win, *v_win;
};

// 16 bytes (piece c) of vertical or window row o
__device__ __forceinline__ void gather_piece(const FreezeParams& p, long head, int o, int c) {
    if (o >= p.k_vl + p.W) return;
    const bool vl = o < p.k_vl;
    // (a vertical index outside [0, N) is clamped: it then names a wrong row instead of memory outside the tensor)
    const int src = vl ? min(max(__ldg(p.idx + head * p.k_vl + o), 0), p.N - 1) : p.N - p.W + (o - p.k_vl);
    const long s = (head * p.N + src) * 16 + c;
    const long d = vl ? (head * p.sK + o) * 16 + c : (head * p.sW + (o - p.k_vl)) * 16 + c;
    (vl ? p.k_vl_out : p.k_win)[d] = __ldg(p.k + s);
    (vl ? p.v_vl_out : p.v_win)[d] = __ldg(p.v + s);
}

template <int G, int FMT>
__global__ void __launch_bounds__(2 * G, FRZ_QTHREADS_PER_SM / (2 * G))
freeze_kernel(const __grid_constant__ FreezeParams p) {
    constexpr int NT = 2 * G;                                  // threads of this CTA
    const int grp = blockIdx.x;
    const long head = blockIdx.y;
    if (grp >= p.n_groups) {
        gather_piece(p, head, (grp - p.n_groups) * (NT / 16) + (threadIdx.x >> 4), threadIdx.x & 15);
        return;
    }
    const int N = p.N, k_vl = p.k_vl, nQ = p.nQ;
    const int32_t* hidx = p.idx + head * k_vl;

    __shared__ int src[G];
    __shared__ uint32_t warp_max[2][NT / 32];
    constexpr bool FMT8 = FMT != HYQ_FMT_INT4;                 // byte-wide codes (INT8 or FP8 e4m3)
    constexpr int ROW_BYTES = FMT8 ? HYQ_D : HYQ_D / 2;        // code bytes per row
    constexpr int TILE_BYTES = 16 * ROW_BYTES;                 // one 16-row V tile
    constexpr float CB = FMT == HYQ_FMT_INT8 ? 127.0f : FMT == HYQ_FMT_FP8_E4M3 ? 448.0f : 7.0f;
    // V codes are staged row-major with 16 bytes of padding per row, so that both the row-wise stores and the
    // word loads of the fragment-major write-out below spread over the banks
    constexpr int VSTRIDE = ROW_BYTES + 16;
    __shared__ __align__(16) uint8_t vstage[G * VSTRIDE];
    // Source rows of the group's G compacted rows in two dependent memory round trips and a short scan: every warp
    // finds j0 = the number of vertical rows before the group's first row by the same 32-way search (no hand-over
    // between warps), then each row walks on from j0 through the few indices that fall inside the group (a row
    // behind a long run of vertical rows falls back to the binary search).
    const int p0 = grp * G;
    int j0;
    {
        const int ln = threadIdx.x & 31;
        int lo = 0, hi = k_vl;                              // smallest j in [lo, hi] with idx[j] - j > p0
        while (lo < hi) {
            const int step = (hi - lo + 31) >> 5;
            const int pos = lo + ln * step;
            const bool below = pos < hi && __ldg(hidx + pos) - pos <= p0;      // predicate still false at pos
            const int f = __popc(__ballot_sync(0xffffffffu, below));            // falses form a prefix of the lanes
            const int new_lo = f ? lo + (f - 1) * step + 1 : lo;
            const int new_hi = f == 0 ? lo : (f < 32 && lo + f * step < hi ? lo + f * step : hi);
            lo = new_lo; hi = new_hi;
        }
        j0 = lo;
    }
    if (threadIdx.x < G) {
        const int row = p0 + threadIdx.x;
        int s = -1;
        if (row < nQ) {
            int j = j0, steps = 0;                          // smallest j >= j0 with idx[j] - j > row
            while (j < k_vl && steps < 16 && __ldg(hidx + j) - j <= row) { ++j; ++steps; }
            s = (steps < 16) ? row + j : source_row(hidx, k_vl, row);
            s = min(s, N - 1);                              // (only a malformed index list can reach the clamp)
        }
        src[threadIdx.x] = s;
    }
    __syncthreads();

    // all loads of both tensors before the first use
    uint4 r[2][4][2];
#pragma unroll
    for (int z = 0; z < 2; ++z) {
        const uint4* x = (z ? p.v : p.k) + head * N * 16;
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {
            const int u = threadIdx.x + gi * NT;              // 16-channel unit: row u >> 3, channels 16 * (u & 7)
            const int s = src[u >> 3];
            r[z][gi][0] = r[z][gi][1] = make_uint4(0, 0, 0, 0);
            if (s >= 0) {
                r[z][gi][0] = __ldg(x + (long)s * 16 + (u & 7) * 2);
                r[z][gi][1] = __ldg(x + (long)s * 16 + (u & 7) * 2 + 1);
            }
        }
    }
    uint32_t mx[2];
#pragma unroll
    for (int z = 0; z < 2; ++z) {
        mx[z] = 0u;
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {
            const uint32_t* w = reinterpret_cast<const uint32_t*>(&r[z][gi][0]);
#pragma unroll
            for (int c = 0; c < 8; ++c) mx[z] = amax_pair(mx[z], w[c]);
        }
        mx[z] = amax_warp(mx[z]);
        if ((threadIdx.x & 31) == 0) warp_max[z][threadIdx.x >> 5] = mx[z];
    }
    __syncthreads();
#pragma unroll
    for (int z = 0; z < 2; ++z) {
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) mx[z] = max(mx[z], warp_max[z][w]);
        const float amax = __uint_as_float(mx[z] << 16);
        const bool dead = !(amax >= 0x1p-100f);
        const float inv = dead ? 0.0f : __fdiv_rn(CB, amax);
        if (threadIdx.x == 0) (z ? p.vs : p.ks)[head * (p.nQp / G) + grp] = dead ? 0.0f : __fdiv_rn(amax, CB);
#pragma unroll
        for (int gi = 0; gi < 4; ++gi) {
            const int u = threadIdx.x + gi * NT;
            const int row = u >> 3, at = (u & 7) * (ROW_BYTES / 8);
            const uint32_t* w = reinterpret_cast<const uint32_t*>(&r[z][gi][0]);
            uint8_t* d = z ? vstage + row * VSTRIDE + at : p.kq + (head * p.nQp + grp * G + row) * ROW_BYTES + at;
            if (FMT == HYQ_FMT_INT8) *reinterpret_cast<uint4*>(d) = quant16_int8(w, inv);
            else if (FMT == HYQ_FMT_FP8_E4M3) *reinterpret_cast<uint4*>(d) = quant16_e4m3(w, inv, dead);
            else *reinterpret_cast<uint2*>(d) = quant16_int4(w, inv);
        }
    }
    {
        // Fragment-major write-out (the layouts of vq_byte_offset / vq8_byte_offset): 16-byte piece number 32 * run + l
        // of a tile, l = 4r + j, is made of one 4-byte load from each of the rows 2j, 2j + 1, 2j + 8, 2j + 9 and
        // a 4 x 4 (INT4) or 2 x 2 (byte codes) transpose of their bytes.
        __syncthreads();
        uint4* dst = reinterpret_cast<uint4*>(p.vq + (head * (p.nQp / 16) + grp * (G / 16)) * (long)TILE_BYTES);
        constexpr int PIECES = TILE_BYTES / 16;
#pragma unroll
        for (int i = 0; i < (G / 16) * PIECES / NT; ++i) {
            const int o = threadIdx.x + i * NT;
            const int tile = o / PIECES, run = (o % PIECES) >> 5, r = (o & 31) >> 2, j = o & 3;
            const int col = FMT8 ? 64 * (run >> 1) + 8 * r + 4 * (run & 1) : 32 * run + 4 * r;
            const uint8_t* base = vstage + (tile * 16 + 2 * j) * VSTRIDE + col;
            const uint32_t e0 = *reinterpret_cast<const uint32_t*>(base);                  // row 2j
            const uint32_t o0 = *reinterpret_cast<const uint32_t*>(base + VSTRIDE);        // row 2j + 1
            const uint32_t e1 = *reinterpret_cast<const uint32_t*>(base + 8 * VSTRIDE);    // row 2j + 8
            const uint32_t o1 = *reinterpret_cast<const uint32_t*>(base + 9 * VSTRIDE);    // row 2j + 9
            uint4 out;
            if (FMT8) {
                out.x = __byte_perm(e0, o0, 0x5140);
                out.y = __byte_perm(e1, o1, 0x5140);
                out.z = __byte_perm(e0, o0, 0x7362);
                out.w = __byte_perm(e1, o1, 0x7362);
            } else {
                const uint32_t t0 = __byte_perm(e0, e1, 0x5140), t1 = __byte_perm(e0, e1, 0x7362);
                const uint32_t t2 = __byte_perm(o0, o1, 0x5140), t3 = __byte_perm(o0, o1, 0x7362);
                out.x = __byte_perm(t0, t2, 0x5410);
                out.y = __byte_perm(t0, t2, 0x7632);
                out.z = __byte_perm(t1, t3, 0x5410);
                out.w = __byte_perm(t1, t3, 0x7632);
            }
            dst[o] = out;
        }
    }
}

// part of a ragged batch's host table of lengths on its way to the device: by value, so that an append needs no copy from
// pageable memory, which waits for the stream (30 us each for the 16 sequences of a step)
constexpr int LENGTH_ROWS = 128, LENGTH_FEW = 32;       // (a launch costs by the size of its parameters, too)
template <int ROWS> struct LengthTable {
    int n;
    int4* dst;
    int4 rows[ROWS];
};

// one new token per sequence: rows [B*Hkv][128] bf16 -> row `row` of every head's staging buffer
template <int ROWS>
__global__ void __launch_bounds__(FRZ_THREADS)
append_rows_kernel(const uint4* __restrict__ k_new, const uint4* __restrict__ v_new, long heads, int row, int Ws,
                   uint4* __restrict__ k_s, uint4* __restrict__ v_s, const __grid_constant__ LengthTable<ROWS> table) {
    pdl_wait();
    pdl_launch_dependents();                 // (the attention that follows waits for this grid's end before it reads anything)
    for (int s = blockIdx.x * FRZ_THREADS + threadIdx.x; s < table.n; s += gridDim.x * FRZ_THREADS) table.dst[s] = table.rows[s];
    const long e = (long)blockIdx.x * FRZ_THREADS + threadIdx.x;     // 16 x 16 bytes per head row
    if (e >= heads * 16) return;
    const long head = e >> 4, c = e & 15;
    const long d = (head * Ws + row) * 16 + c;
    k_s[d] = __ldg(k_new + e);
    v_s[d] = __ldg(v_new + e);
}

template <int ROWS>
static int launch_append(const void* k_new, const void* v_new, long heads, int row, int Ws, void* k_s, void* v_s,
                         const LengthTable<ROWS>& table, cudaStream_t st) {
    return launch_pdl(append_rows_kernel<ROWS>, dim3((unsigned)((heads * 16 + FRZ_THREADS - 1) / FRZ_THREADS)), dim3(FRZ_THREADS), 0, st,
                      static_cast<const uint4*>(k_new), static_cast<const uint4*>(v_new), heads, row, Ws, static_cast<uint4*>(k_s),
                      static_cast<uint4*>(v_s), table);
}

int launch_cache_append(const void* k_new, const void* v_new, const hyq_kv_cache& c, cudaStream_t st) {
    LengthTable<1> none{};
    return launch_append(k_new, v_new, (long)c.B * c.Hkv, c.n_staging, c.staging_capacity, c.k_s, c.v_s, none, st);
}

template <int ROWS>
static int launch_append_ragged(const void* k_new, const void* v_new, const hyq_kv_cache& c, int b, const int32_t* lengths_host,
                                int row, int32_t* lengths, cudaStream_t st) {
    const size_t at = (size_t)b * c.Hkv * c.staging_capacity * HYQ_D * 2;
    int rc = HYQ_OK;
    for (int s0 = 0; s0 < c.B && rc == HYQ_OK; s0 += ROWS) {    // (the rows themselves with every part of the table)
        LengthTable<ROWS> t;
        t.n = c.B - s0 < ROWS ? c.B - s0 : ROWS;
        t.dst = reinterpret_cast<int4*>(lengths) + s0;
        memcpy(t.rows, lengths_host + 4 * s0, (size_t)t.n * sizeof(int4));
        if (b >= s0 && b < s0 + t.n) t.rows[b - s0].w = row + 1;
        rc = launch_append(k_new, v_new, c.Hkv, row, c.staging_capacity, static_cast<char*>(c.k_s) + at, static_cast<char*>(c.v_s) + at, t, st);
    }
    return rc;
}

int launch_cache_append_ragged(const void* k_new, const void* v_new, const hyq_kv_cache& c, int b, const int32_t* lengths_host,
                               int row, int32_t* lengths, cudaStream_t st) {
    return c.B <= LENGTH_FEW ? launch_append_ragged<LENGTH_FEW>(k_new, v_new, c, b, lengths_host, row, lengths, st)
                             : launch_append_ragged<LENGTH_ROWS>(k_new, v_new, c, b, lengths_host, row, lengths, st);
}

int launch_freeze(const void* k_, const void* v, const int32_t* vl_idx, const hyq_kv_cache& c, cudaStream_t st) {
    const CacheGeo g = cache_geo(c);
    const long heads = (long)c.B * c.Hkv;
    FreezeParams p;
    p.k = static_cast<const uint4*>(k_); p.v = static_cast<const uint4*>(v); p.idx = vl_idx;
    p.N = c.N; p.W = g.W; p.k_vl = c.k; p.nQ = (int)g.nQ; p.n_groups = (int)(g.nQp / c.group);
    p.nQp = g.sQ; p.sK = g.sK; p.sW = g.sW;
    p.kq = static_cast<uint8_t*>(c.kq_codes); p.vq = static_cast<uint8_t*>(c.vq_codes);
    p.ks = c.kq_scales; p.vs = c.vq_scales;
    p.k_vl_out = static_cast<uint4*>(c.k_vl); p.v_vl_out = static_cast<uint4*>(c.v_vl);
    p.k_win = static_cast<uint4*>(c.k_win); p.v_win = static_cast<uint4*>(c.v_win);
    const int rows = 2 * c.group / 16;                          // rows a gathering block copies
    const dim3 grid((unsigned)(p.n_groups + (c.k + g.W + rows - 1) / rows), (unsigned)heads);
    if (grid.x == 0) return HYQ_OK;
#define HYQ_FRZ(G_, F_) freeze_kernel<G_, F_><<<grid, 2 * G_, 0, st>>>(p)
#define HYQ_FRZ_F(G_) do { if (c.format == HYQ_FMT_INT8) HYQ_FRZ(G_, HYQ_FMT_INT8); else if (c.format == HYQ_FMT_FP8_E4M3) HYQ_FRZ(G_, HYQ_FMT_FP8_E4M3); else HYQ_FRZ(G_, HYQ_FMT_INT4); } while (0)
    if (c.group == 32) HYQ_FRZ_F(32);
    else if (c.group == 64) HYQ_FRZ_F(64);
    else HYQ_FRZ_F(128);
#undef HYQ_FRZ_F
#undef HYQ_FRZ
    return launch_status();
}

}  // namespace hyq

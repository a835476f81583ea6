// Declarations shared by the attention pre-pass and the attention kernels.
#pragma once
#include "common.cuh"

namespace hyq {

// number of query rows of a call (the query block may be shorter than the keys; 0 means "all L")
__host__ __device__ inline int query_rows(const hyq_attn_args& a) { return a.Lq > 0 ? a.Lq : a.L; }

constexpr int TC_ROWS = 256;                // query rows of a work unit (two 128-row tiles of one query head)
constexpr int TC_SMS = 148;
constexpr int VL_TILE_BYTES = 1024;
// element 0 of a key's row in the vertical-line operand: e4m3 scores get -inf in e5m2 added for a vertical-line key (0 otherwise);
// integer scores start from 2^63 times a bf16 number, 1.5 * 2^23 or, for a vertical-line key, -1.5 * 2^127 (attn_tc.cu, LIFT)
constexpr uint32_t VL_KNOCK_E5M2 = 0xFCu, VL_KNOCK_BF16 = 0xDFC0u, VL_PLAIN_BF16 = 0x2BC0u;
constexpr int TC_MAX_SEQ = 32;              // sequences of one ragged launch (the table travels as a kernel parameter) ...
constexpr int TC_MAX_LEVELS = 512;          // ... and units per head of its longest sequence

// One sequence of a launch.  A plain call is one sequence with B * Hq heads; a ragged call has one entry per prompt.
// Rows are counted in the flattened [heads * rows] views of the buffers: row i of head h of the sequence is row
// q_row0 + h * Lq + i of Q, kv_row0 + (h / g) * L + j of K and V, vl_row0 + h * k + j of the gathered rows.
struct TcSeq {
    int L, Lq, k;
    int q_row0, kv_row0, vl_row0;
    int qs0, ks0;                           // first entry in q_scales / k_scales (and v_scales)
    int nb, nbq;                            // quantization blocks per head of the keys / the query block
    int mask_words, mask0;                  // bitmask words per head (a multiple of 4), first word of the sequence
    int levels;                             // units per head
    int split;                              // CTAs that share the sequence's units tile by tile (0: one CTA per unit)
    int cta0, slot0;                        // split: first CTA behind the unsplit units, first slot for partial results ...
    int src;                                // the sequence's number in the caller's order
    int tiles;                              // ... and key tiles of all its units together (as tc_unit_tiles counts them),
    int lead;                               // each unit counted `lead` tiles longer than it is: the cost of beginning it
};

struct TcSeqTable {
    int n_seq, heads, g;                    // heads: query heads per sequence; g: of them per KV head
    int n_unsplit;                          // sequences 0 .. n_unsplit-1 run one CTA per unit, most units per head first
    int unsplit_ctas, ctas;                 // grid: the unsplit units, then the split sequences' CTAs
    int kv_rows, vl_rows, q_rows;           // totals of the flattened views
    TcSeq seq[TC_MAX_SEQ];
};
// unsplit units before level l, level 0 being the longest (only consulted when more than one sequence is unsplit)
struct TcLevels {
    int cum[TC_MAX_LEVELS];
};
struct TcTables {                           // what a launch that is not a plain whole prefill needs to find its work
    TcSeqTable tab;
    TcLevels lev;
};

// Key tiles a unit can have at most: low-bit, vertical-line and window tiles of its 256 rows at positions a0 .. a1
// (the vertical tiles bounded by k, so that the host can know the number).
__host__ __device__ inline int tc_unit_tiles(int L, int Lq, int k, int window, int fixed_tail, int unit) {
    const int i1 = (unit * TC_ROWS + TC_ROWS - 1 < Lq - 1) ? unit * TC_ROWS + TC_ROWS - 1 : Lq - 1;
    const int a0 = L - Lq + unit * TC_ROWS, a1 = L - Lq + i1;
    const int lim = L - window - 1;
    const int h0 = fixed_tail ? (a0 < lim ? a0 : lim) : a0 - window, h1 = fixed_tail ? (a1 < lim ? a1 : lim) : a1 - window;
    const int nA = h1 >= 0 ? h1 / 64 + 1 : 0, kk = k < h1 + 1 ? k : h1 + 1, nB = kk > 0 ? (kk + 63) / 64 : 0;
    const int c0 = (h0 + 1 > 0 ? h0 + 1 : 0) / 64;
    return nA + nB + (window > 0 ? a1 / 64 - c0 + 1 : 0);
}

// byte offsets into the caller's workspace (tensor-core kernel)
struct TcWorkspace {
    size_t vl_bits;     // uint32 [heads][mask_words] per sequence: vertical-line bitmask over key positions
    size_t v16;         // fp16 [kv_rows][D]            V
    size_t vh16;        // fp16 [kv_rows][D]            V^ without the mantissa of its scale: code * 2^e (value_factor)
    size_t kv_fac;      // f32x4, a block each          K scale, log2 of that mantissa and its reciprocal
    size_t kvl;         // bf16 [vl_rows][D]            gathered vertical-line K rows
    size_t vvl;         // fp16 [vl_rows][D]            gathered vertical-line V rows
    size_t q8;          // u8   [q_rows][D]             INT4 only: Q codes as e4m3 bytes
    size_t k8;          // u8   [kv_rows][D]            INT4 only: K codes as e4m3 bytes
    size_t vl_tiles;    // u8   [mask_words/2][1024] per head: the first 16 bytes of every key's row of the vertical-line operand
                        //                              (element 0 as above, zero elsewhere), [64 keys][16 bytes] per tile
    size_t redo;        // i32x4 [1 + pieces]           pieces of work the second launch does again, behind their count
    size_t part_o;      // f32  [slots][256][D]         split sequences only: partial accumulators ...
    size_t part_ml;     // f32  [slots][256][2]         ... and (reference maximum, row sum) per row
    size_t total;
    int mask_words;     // bitmask words of all heads and sequences
    int slots;          // partial results
    int pieces;         // pieces of work at most (entries of the redo list)
};

// e4m3 scores need the vertical-line operand only where there are vertical-line keys; integer scores are lifted by it
inline bool tc_has_vl_tiles(const hyq_attn_args& a, long vl_rows) { return a.q_format == HYQ_FMT_INT8 || vl_rows > 0; }

struct TcPlan {
    TcTables t;
    TcWorkspace w;
};

// Fills the plan of a launch.  seq[0 .. n_seq): the sequences' L, Lq, k and offsets into the caller's buffers (q_row0,
// kv_row0, vl_row0, qs0, ks0); everything else is derived.  Returns false when the table cannot hold the launch.
bool tc_make_plan(const hyq_attn_args& a, const TcSeq* seq, int n_seq, int heads, int g, TcPlan& plan);
// the plan of a plain call
bool tc_plain_plan(const hyq_attn_args& a, TcPlan& plan);
// workspace for a plain call and for any smaller one
size_t tc_query_bytes(const TcPlan& plan);
// one sequence of a ragged call as tc_make_plan takes it; Hq / Hkv times the tokens, vertical keys and blocks before it
TcSeq tc_ragged_seq(const hyq_attn_args& a, int L, int k, size_t tokens_before, size_t k_before, size_t nb_before);

// A call that quantizes and attends in one: Q, K, V per sequence wherever they lie (in the caller's order), and the pre-pass's
// fp16 values and widened codes already written by the quantizer.
struct TcSources {
    const void *q[TC_MAX_SEQ], *k[TC_MAX_SEQ], *v[TC_MAX_SEQ];
};
int launch_tc_prepass(const hyq_attn_args& a, const TcPlan& plan, const TcSources* src, cudaStream_t st);
// the whole tensor-core attention of a planned call (64-token quantization blocks / the others); src: see there, may be null
int launch_attn_tc(const hyq_attn_args& a, const TcPlan& plan, const TcSources* src, float alpha, cudaStream_t st);
namespace tcbt {
int launch_attn_tc(const hyq_attn_args& a, const TcPlan& plan, const TcSources* src, float alpha, cudaStream_t st);
}

// Test hooks of the tensor-core kernel (hyq_test_set_attention_hooks): the clock limit of a single barrier wait
// (0: the default of about two seconds) and the walk position whose K/V load the producer leaves out (-1: none).
struct TcTestHooks {
    long long wait_limit;
    int drop_load;
};
TcTestHooks tc_test_hooks();

// zero-fills bits[n_heads][mask_words] and sets one bit per vertical-line key (memset + one kernel)
int launch_vl_bitmask(const int32_t* idx, long n_heads, int k, int L, int mask_words, uint32_t* bits, cudaStream_t st);

}  // namespace hyq

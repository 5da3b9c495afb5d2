// Staged mixed-precision GEMM / implicit-GEMM convolution on the sm_103a
// tensor cores: expand the packed codes once into tensor-pipe operands in
// caller scratch, then run a persistent tcgen05 GEMM over them.
//
// What it computes (Sec. 3 "Enabling Low-Cost Fixed-Point Operations";
// Sec. 4.2): for each precision group g the exact integer dot products
//   Acc_g[m][n] = sum over k in group g of u[m][k] * j[n][k]
// and Y = sum_g s_a * s_w * Acc_g / ((2^na - 1) * 2^(nw - 1)) in fp32.
//
// Why staged.  Expanding packed codes inside the GEMM tiles (the fused
// kernel of mma_gemm.cu) repeats the expansion of every activation row once
// per column tile and of every weight row once per row tile, and that work,
// not the tensor pipe, sets its speed.  Here each code is expanded exactly
// once, by a streaming kernel, into a byte layout the MMA reads directly;
// the expanded operands (e.g. 63 MB for an 8192 x 4096 x 4096 layer) stay
// in the 129 MB L2 while the GEMM reads them.
//
// Operand encodings (all exact; one group at a time along K):
//   * groups with <= 4-bit codes on both sides: E4M3 bytes.  An activation
//     code u < 16 as a raw byte is the E4M3 value u * 2^-9; a weight code j in
//     [-8, 7] is stored sign-magnitude, the E4M3 value j * 2^-9.  The fp32
//     accumulator holds sum u*j * 2^-18 exactly (|sum| <= 65536 * 15 * 8 <
//     2^24), so the epilogue scales by 2^18.
//   * wider groups: fp16.  Activations are centred, u - 2^(na-1) (padding and
//     taps outside the image count as u = 0), weights are j; every product
//     and partial sum is an integer.  The epilogue adds back
//     2^(na-1) * C[n] with C[n] the weight row's code sum (from the expander).
//     A partial sum stays exact while |sum| <= 2^24; a group whose worst case
//     over its K range could exceed that is accumulated in segments that the
//     epilogue warps drain into int32 registers.
//
// The GEMM kernel: persistent CTAs (one per SM) walk output tiles of 128 rows by
// 256 columns (240, 128 or 64 where that fits the layout or the shape better;
// pairs of CTAs: 256 x 256, or 240).
//   warp 0      TMA producer: per 128-byte K-stage, an A box (128 rows, 16 KB)
//               and a B box, 128-byte swizzle, a ring as deep as shared memory allows
//   warp 1      TMEM owner and MMA issuer: 4 MMAs per K-stage.
//               A tile's accumulation is a sequence of jobs (a group, one
//               exact segment of a group, or one scale run; the segmented group first), and job
//               k of the CTA accumulates into TMEM region k % 2 (256 columns
//               each), so the epilogue drains one region while the MMAs fill
//               the other, across tile boundaries too
//   warps 4-11  epilogue: two warps per TMEM lane quadrant, half of the tile's
//               columns each; earlier jobs of a tile are kept in registers,
//               the final job completes the outputs
// The issuing warps run their loops with all lanes and put only the TMA and MMA
// instructions under an elected lane, so that descriptors and addresses stay in
// uniform registers: under `lane == 0` each 4-MMA stage took 600-640 cycles to
// issue, whatever the tile's width, where the pair's MMAs take 512 (the
// 8192 x 4096 x 4096 4/8-bit call went from 121 to 109 us with this alone; its
// MMAs without loads or epilogue take 75 us, and the operand expansion 22).
// Every wait is bounded (2 s); a wait that runs out records an error bit,
// raises a CTA abort flag and the CTA winds down (copies and MMAs in flight
// are waited for, TMEM is freed).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstring>
#include <type_traits>

#include "packed_words.cuh"
#include "soniq_device.cuh"
#include "soniq_internal.h"
#include "tc_ptx.cuh"

namespace soniq {
namespace staged {

using namespace tc;

constexpr int BM = 128;
constexpr int BN = 256;                              // tile width (layouts without E2M1 groups)
constexpr int BN_F4 = 240;                           // tile width of layouts with E2M1 groups
constexpr int REGION = 256;                          // TMEM columns per accumulator region
constexpr int SF_COLS = 16;                          // E2M1 scale factors: region columns BN_F4 .. +15
constexpr int KSTAGE = 128;                          // bytes of K per ring stage (128-byte swizzle)
constexpr int A_BYTES = BM * KSTAGE;
constexpr int NUM_EPI_WARPS = 8;
constexpr int WARP_TMA = 0, WARP_MMA = 1, WARP_EPI = 4;      // warps 2 and 3 only give up registers
constexpr int NUM_THREADS = (WARP_EPI + NUM_EPI_WARPS) * 32;

// Epilogues.  LEAN, SEG, NEXT, NEXT_SEG and RUNS read the accumulators as MMA fragments
// (fragment epilogue below); GENERAL and GENERAL_NEXT, one row per lane, also
// write debug accumulators.
enum {
    EPI_LEAN = 0,          // both groups accumulated in one piece each
    EPI_SEG = 1,           // one group in exact segments, drained to int32
    EPI_NEXT = 2,          // LEAN, plus the next layer's codes (quantize-in-epilogue)
    EPI_RUNS = 3,          // scale runs along K
    EPI_NEXT_SEG = 4,      // NEXT with one group in exact segments (us, GENERAL_NEXT and this: 16384 x 2304 x 512
                           // at 8 bits 121, 66.5; 2048 x 4096 x 4096 123, 77; 253 x 1856 x 4224 44, 29)
    EPI_GENERAL = 5,
    EPI_GENERAL_NEXT = 6
};

template <int EPI>
constexpr bool kEpiSegments = EPI == EPI_SEG || EPI == EPI_NEXT_SEG;
template <int EPI>
constexpr bool kEpiNext = EPI == EPI_NEXT || EPI == EPI_NEXT_SEG;

// How outputs leave: OUT_BATCH stages 32 rows x 32 columns per epilogue warp
// (2 KB) at a time and copies them out with 16-byte stores, which leaves the
// shared memory to the operand ring (six 32 KB stages for a pair); OUT_TMA
// stages a warp's whole tile (8 KB) for TMA stores, the quicker epilogue where
// few K-stages per tile leave it on the critical path.  GEMM calls, batch
// against TMA: 8192 x 4096 x 4096 4/8 bits (40 K-stages, pairs) 121 and 125 us, its
// 2/8-bit layout with E2M1 groups 97 and 108 us, 16384 x 768 x 3072 (9 K-stages)
// 75 and 69 us.
enum { OUT_BATCH = 0, OUT_TMA = 1, OUT_GENERAL = 2 };

// Shared memory of a variant: the operand ring, the epilogue warps' output
// staging, the tile's column constants (16 bytes per column, two tiles' worth;
// GENERAL: one copy per warp), the barriers, misc words (tmem base, abort flag,
// a zero word).
template <int BNT, bool PAIR, int OUT>
struct Cfg {
    static constexpr int B_BYTES = (PAIR ? BNT / 2 : BNT) * KSTAGE;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = (OUT == OUT_BATCH ? 192 : 144) * 1024 / STAGE_BYTES;
    static constexpr int EPI_COLS = BNT / (NUM_EPI_WARPS / 4);
    static constexpr int COLS_BYTES = EPI_COLS * 16;               // constants of one warp's columns
    static constexpr int OUT_PER_WARP = OUT != OUT_BATCH ? (32 * EPI_COLS * 2 + 1023) / 1024 * 1024 : 2048;
    static constexpr int BAR_FULL = 0, BAR_EMPTY = STAGES, BAR_REG_FULL = 2 * STAGES, BAR_REG_EMPTY = 2 * STAGES + 2,
                         BAR_TEARDOWN = 2 * STAGES + 4, BAR_COLS = 2 * STAGES + 5, NUM_BARS = 2 * STAGES + 9;
    static constexpr int SMEM_OUT = STAGES * STAGE_BYTES;
    static constexpr int SMEM_COLS = SMEM_OUT + NUM_EPI_WARPS * OUT_PER_WARP;
    static constexpr int SMEM_BAR = SMEM_COLS + 8 * COLS_BYTES;
    static constexpr int SMEM_MISC = SMEM_BAR + NUM_BARS * 8;
    static constexpr int SMEM_ALLOC = SMEM_MISC + 16 + 1024;      // slack for 1024-byte alignment
    static_assert(SMEM_ALLOC <= 227 * 1024, "the ring and the epilogue's buffers fit");
};
constexpr long long kTimeoutNs = 2000000000LL;

struct SGroup {
    int32_t kind;          // 0: E4M3 bytes, 1: fp16, 2: E2M1 nibbles (kind::mxf4)
    int32_t stages;        // 128-byte K-stages of the group
    int32_t x0;            // byte offset of the group in an expanded row
    int32_t seg_stages;    // K-stages per exact segment (segmented group only)
    int32_t n_seg;         // segments (1: accumulated in one piece)
    int32_t center;        // fp16 activations carry -center; the epilogue adds center * C[n]
    float acc_scale;       // 2^18 (E4M3), 1 (fp16) or 4 (E2M1)
    float inv_levels;      // 1 / ((2^na - 1) * 2^(nw - 1))
};

struct SParams {
    CUtensorMap tma_a;     // expanded activations [rows][eb]
    CUtensorMap tma_b;     // expanded weights [N][eb] (each CTA of a pair loads half the tile's rows)
    CUtensorMap tma_y;     // outputs [M][N] (2-byte elements), 64 x 32 boxes, when y_tma
    const float* s_a;
    const float* s_w;
    const int32_t* colsum; // [N][2] weight code sums
    void* Y;
    int32_t* acc_dbg;
    unsigned* err;
    int64_t M;
    int32_t N;
    int32_t m_tiles, n_tiles, total_tiles;
    int32_t pair_tiles;    // CTA pairs: (m tile pair, n tile) units, m tile pairs = ceil(m_tiles / 2)
    int32_t s_a_per_row;
    int32_t out_bf16;
    int32_t seg_group;     // group accumulated in drained segments, or -1
    int32_t drop_first;    // test hook: the producer never issues the first K-stage
    int32_t y_tma;         // 1: outputs leave through shared memory and TMA stores
    int32_t write_y;       // 0: Y is not written (only the next layer's codes)
    // quantize-in-epilogue: output column j is packed position j of the next layer
    int32_t has_next;
    const float* s_next;   // the next layer's calibrated activation scales [2]
    uint8_t* Ap_next;      // its packed activation rows
    int32_t next_row_bytes;
    int32_t next_pa0;      // first packed position of its group 1
    int32_t next_count[2], next_bits[2], next_off[2];
    // scale runs along K: every job is one run of one group, scaled on its own;
    // s_a is [rows or 1][2][nb], s_w [N][2][nb]
    int32_t runs, nb;
    SGroup g[2];
};

// ---------------------------------------------------------------------------
// Expansion of packed rows into tensor-pipe operands
// ---------------------------------------------------------------------------

struct ExpandParams {
    const uint8_t* src;        // packed rows
    int64_t src_row_bytes;
    uint8_t* dst;              // expanded rows
    int64_t dst_row_bytes;
    int32_t* colsum;           // weights: [rows][2] code sums of fp16 groups (else unused)
    int64_t rows;              // output rows (conv activations: output pixels)
    int32_t is_weight;
    int32_t bits[2], kind[2], src_off[2], dst_off[2], blk_src[2], blk_dst[2], center[2];
    // implicit-GEMM convolution (activations): block kb of group g is tap kb / cpt[g],
    // channel block kb % cpt[g] of the input pixel that tap reads
    int32_t conv, H, W, P, Q, R, S, sh, sw, ph, pw;
    int32_t cpt[2];
    uint64_t cpt_magic[2];     // ceil(2^32 / cpt): tap = (kb * magic) >> 32, exact for kb < 2^32 / cpt
    int32_t vec8[2];           // source blocks of the group can be read as 8-byte vectors
    // code encoding of each group: 0 unsigned, 1 n-bit two's complement (weights,
    // signed activations), 2 one-bit +-1 (bit 1 -> +1, bit 0 -> -1, positions
    // from count[g] on -> 0)
    int32_t code_kind[2], count[2];
};

// n-bit two's-complement patterns in the bytes of x -> E4M3 sign-magnitude bytes.
template <int N>
__device__ __forceinline__ uint32_t twos_to_e4m3(uint32_t x) {
    const uint32_t neg = ((x >> (N - 1)) & 0x01010101u) * 0xFFu;   // 0xFF in negative bytes
    const uint32_t mag = ((1u << N) * 0x01010101u) - x;           // 2^N - x per byte, no borrow (x < 2^N)
    return (x & ~neg) | ((mag | 0x80808080u) & neg);
}

// 16 bytes of operands from the words of part `part` of block kb (of group g).
template <int N, int PARTS>
__device__ __forceinline__ uint4 encode_piece(const ExpandParams& p, const PartWords<N, PARTS>& w, int g, int ck, int kb,
                                              int part, __half2 bias, int32_t& csum) {
    uint32_t o[PartWords<N, PARTS>::TW];
    w.bytes(part, o);
    if constexpr (PARTS == 1) {
        // E2M1, two codes per byte (the first in the low nibble): a code c with
        // |c| <= 4 is sign << 3 | |c|, the value c / 2
        uint32_t y[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            uint32_t x = o[t];
            if (ck == 1) {
                // two's complement to sign << 3 | |c|: of one bit, 1 is -1; of two, 01 is 1, 11 -1, 10 -2
                if constexpr (N == 1) x |= x << 3;
                else x = ((x << 2) & 0x08080808u) | (x & ~(x << 1) & 0x02020202u) | (x & 0x01010101u);
            }
            y[t] = x | (x >> 4);                                        // bytes 0 and 2: two codes each
        }
        return make_uint4(__byte_perm(y[0], y[1], 0x6420u), __byte_perm(y[2], y[3], 0x6420u),
                          __byte_perm(y[4], y[5], 0x6420u), __byte_perm(y[6], y[7], 0x6420u));
    } else if constexpr (PARTS == 2) {
        if (ck == 1) {
#pragma unroll
            for (int t = 0; t < 4; ++t) o[t] = twos_to_e4m3<N>(o[t]);
        } else if (ck == 2) {
            // one-bit +-1: bit 1 -> E4M3 +2^-9 (0x01), bit 0 -> -2^-9 (0x81); none past count
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int valid = p.count[g] - (kb * 32 + 16 * part + 4 * t);
                const uint32_t keep = valid >= 4 ? 0xFFFFFFFFu : (valid <= 0 ? 0u : (1u << (8 * valid)) - 1u);
                o[t] = (0x81818181u - (o[t] & 0x01010101u) * 0x80u) & keep;
            }
        }
        return make_uint4(o[0], o[1], o[2], o[3]);
    } else {
        uint32_t h[4];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            // signed codes: offset binary j + 2^(n-1); unsigned: the code u
            const uint32_t x = ck == 1 ? (o[t] ^ (0x01010101u << (N - 1))) : o[t];
            if (p.is_weight) csum += (int32_t)__dp4a(x, 0x01010101u, 0u);
            uint32_t lo, hi;
            bytes_to_magic_half2(x, lo, hi);
            h[2 * t] = half2_sub(lo, bias);
            h[2 * t + 1] = half2_sub(hi, bias);
        }
        return make_uint4(h[0], h[1], h[2], h[3]);
    }
}

constexpr int kExpandRows = 4;      // rows a warp expands together

// Rows r0 .. r0 + 3 (as far as they exist) of group g, by one warp; one
// 16-byte piece of an expanded row per lane.
//
// Bound by L2 traffic (each packed byte read, each operand byte written once)
// and by the latency of the loads.  A lane forms 16 output bytes (16 codes of
// E4M3, 8 of fp16, 32 of E2M1) from the words that hold them, so every store
// instruction writes 512 contiguous bytes; a whole block per lane wrote each
// 32-byte sector in two instructions.  Four rows keep that many independent
// loads in flight and share the index arithmetic.  Convolutions (64 x 56 x 56 x 64, 3 x 3,
// 282 MB of operands: 192 us a call with one row per warp, 155 with four; 64 x 14 x 14 x 256
// 29.7 and 29.2; their weights' rows in the same launch).
template <int N, int PARTS>
__device__ __forceinline__ void expand_rows(const ExpandParams& p, int64_t r0, int g, int lane) {
    using Words = PartWords<N, PARTS>;
    constexpr int TW = Words::TW;
    const bool vec8 = p.vec8[g] != 0;
    const int ck = p.code_kind[g];
    const int nr = (int)(p.rows - r0 < kExpandRows ? p.rows - r0 : kExpandRows);
    uint8_t* drow = p.dst + r0 * p.dst_row_bytes + p.dst_off[g];
    const uint8_t* srow[kExpandRows];     // the row's group (conv: its image's)
    int hp[kExpandRows], wq[kExpandRows];
#pragma unroll
    for (int i = 0; i < kExpandRows; ++i) {
        const int64_t r = r0 + (i < nr ? i : 0);
        hp[i] = wq[i] = 0;
        if (!p.conv) {
            srow[i] = p.src + r * p.src_row_bytes + p.src_off[g];
        } else {
            const uint32_t pq = (uint32_t)p.P * (uint32_t)p.Q, ru = (uint32_t)r;      // rows < 2^31
            const uint32_t img = ru / pq, rem = ru - img * pq, pp = rem / (uint32_t)p.Q;
            hp[i] = (int)pp * p.sh - p.ph;
            wq[i] = (int)(rem - pp * (uint32_t)p.Q) * p.sw - p.pw;
            srow[i] = p.src + (int64_t)img * p.H * p.W * p.src_row_bytes + p.src_off[g];
        }
    }
    const __half2 bias = __half2half2(__ushort_as_half(
        (unsigned short)(0x6400u + (ck == 1 ? (1u << (N - 1)) : (uint32_t)p.center[g]))));
    int32_t csum[kExpandRows];
#pragma unroll
    for (int i = 0; i < kExpandRows; ++i) csum[i] = 0;
    const int pieces = p.blk_dst[g] * PARTS;
    for (int c = lane; c < pieces; c += 32) {
        const int kb = c / PARTS, part = c % PARTS;
        Words w[kExpandRows];
        if (!p.conv) {
            const bool in = kb < p.blk_src[g];
#pragma unroll
            for (int i = 0; i < kExpandRows; ++i) {
                if (in) w[i].load(GlobalWords(srow[i] + kb * 4 * N), part, vec8);
                else w[i].zero();
            }
        } else {
            const int tap = (int)(((uint64_t)kb * p.cpt_magic[g]) >> 32);
            const int cb = kb - tap * p.cpt[g];
            const int rr = tap / p.S, ss = tap - rr * p.S;
            const bool in = tap < p.R * p.S;
#pragma unroll
            for (int i = 0; i < kExpandRows; ++i) {
                const int h = hp[i] + rr, x = wq[i] + ss;
                if (in && h >= 0 && h < p.H && x >= 0 && x < p.W)
                    w[i].load(GlobalWords(srow[i] + ((int64_t)h * p.W + x) * p.src_row_bytes + cb * 4 * N), part,
                              vec8);
                else
                    w[i].zero();
            }
        }
#pragma unroll
        for (int i = 0; i < kExpandRows; ++i) {
            const uint4 d = encode_piece<N, PARTS>(p, w[i], g, ck, kb, part, bias, csum[i]);
            if (i < nr) *reinterpret_cast<uint4*>(drow + i * p.dst_row_bytes + (int64_t)c * 16) = d;
        }
    }
    if (PARTS == 4 && p.is_weight) {
        // sum of j over the row's group: the offset-binary sum minus 2^(n-1) per code
#pragma unroll
        for (int i = 0; i < kExpandRows; ++i) {
            const int32_t s = __reduce_add_sync(0xffffffffu, csum[i]);
            if (lane == 0 && i < nr) p.colsum[(r0 + i) * 2 + g] = s - (1 << (N - 1)) * 32 * p.blk_dst[g];
        }
    }
}

// Item `it` (rows 4 (it / 2) .. + 3, group it % 2) of one operand.
__device__ __forceinline__ void expand_item(const ExpandParams& p, int64_t it, int lane) {
    const int64_t r = (it >> 1) * kExpandRows;
    const int g = (int)(it & 1);
    if (p.blk_dst[g] == 0) return;
    if (p.kind[g] == 2) {
        if (p.bits[g] == 1) expand_rows<1, 1>(p, r, g, lane);
        else expand_rows<2, 1>(p, r, g, lane);
    } else if (p.kind[g] == 0) {
        switch (p.bits[g]) {
            case 1: expand_rows<1, 2>(p, r, g, lane); break;
            case 2: expand_rows<2, 2>(p, r, g, lane); break;
            case 3: expand_rows<3, 2>(p, r, g, lane); break;
            default: expand_rows<4, 2>(p, r, g, lane); break;
        }
    } else {
        switch (p.bits[g]) {
            case 1: expand_rows<1, 4>(p, r, g, lane); break;
            case 2: expand_rows<2, 4>(p, r, g, lane); break;
            case 3: expand_rows<3, 4>(p, r, g, lane); break;
            case 4: expand_rows<4, 4>(p, r, g, lane); break;
            case 5: expand_rows<5, 4>(p, r, g, lane); break;
            case 6: expand_rows<6, 4>(p, r, g, lane); break;
            case 7: expand_rows<7, 4>(p, r, g, lane); break;
            default: expand_rows<8, 4>(p, r, g, lane); break;
        }
    }
}

// Both operands in one launch: items 0 .. items(pa) - 1 are (four rows, group)
// of the activations, the rest of the weights (pw).
__global__ void __launch_bounds__(256, 4) expand_kernel(const __grid_constant__ ExpandParams pa,
                                                     const __grid_constant__ ExpandParams pw) {
    tc::pdl_wait();   // launched with launch_pdl: the packed rows are written before this
    const int lane = threadIdx.x & 31;
    const int64_t warp_id = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t items_a = (pa.rows + kExpandRows - 1) / kExpandRows * 2;
    const int64_t items = items_a + (pw.rows + kExpandRows - 1) / kExpandRows * 2;
    for (int64_t item = warp_id; item < items; item += nwarps) {
        if (item < items_a) expand_item(pa, item, lane);
        else expand_item(pw, item - items_a, lane);
    }
}

// The same for a linear layer, from packed rows staged in shared memory.
//
// With loads straight from global memory (expand_kernel) a warp waits for L2
// once per 32 pieces, and the short kernel's straight-line code is fetched
// cold: 20 us for the 8192 x 4096 x 4096 4/8-bit layer (94 MB moved), most stalls on
// loads and on instruction fetch; streamed, 13 us.  Here a producer warp
// streams tiles of packed rows (contiguous, so one bulk copy each)
// through a ring; each consumer warp expands one row of a tile, two pieces per
// step, with a short loop per group, and stores 512 contiguous bytes at a time.
// Rows of which eight do not fit twice are shared by two, four or eight warps, whose
// code sums meet in shared memory; the producer writes them out when it takes the
// stage back (8 bits, calls in us, from global memory and streamed: 1000 x 60000 x 64
// 457, 259; 137 x 11008 x 11008 173, 128; 4096 x 7000 x 1024 86, 69).
constexpr int kStreamWarps = 8;             // consumers
constexpr int kStreamMaxStages = 6;
constexpr size_t kStreamSmemPerSm = 216 * 1024;

struct StreamParams {
    ExpandParams op[2];       // activations, weights
    unsigned* err;
    int32_t stages, stage_bytes;
    int32_t rpw;              // rows of a tile per warp
    int32_t wpr;              // warps per row (1, 2, 4 or 8; rpw is 1 above 1)
};

// One group of nr staged rows (row r's packed codes at src), by one warp of wpr: its
// pieces are those of index sub modulo wpr, 32 at a time.  sum: wpr > 1, the shared
// word of the row's and group's code sum.
template <int N, int PARTS, bool LONG>
__device__ __forceinline__ void stream_group(const ExpandParams& p, uint32_t src, int64_t r, int nr, int g, int lane, int sub,
                                             int wpr, int32_t* sum) {
    const bool vec8 = p.vec8[g] != 0;
    const int ck = p.code_kind[g];
    const __half2 bias = __half2half2(__ushort_as_half(
        (unsigned short)(0x6400u + (ck == 1 ? (1u << (N - 1)) : (uint32_t)p.center[g]))));
    uint8_t* drow = p.dst + r * p.dst_row_bytes + p.dst_off[g];
    const int pieces = p.blk_dst[g] * PARTS, have = p.blk_src[g] * PARTS;
#pragma unroll 1
    for (int i = 0; i < nr; ++i, src += (uint32_t)p.src_row_bytes, drow += p.dst_row_bytes) {
        int32_t csum = 0;
#pragma unroll 2
        for (int c = LONG ? lane + 32 * sub : lane; c < pieces; c += LONG ? 32 * wpr : 32) {
            const int kb = c / PARTS, part = c % PARTS;
            PartWords<N, PARTS> w;
            if (c < have) w.load(SharedWords{src + (uint32_t)(kb * 4 * N)}, part, vec8);
            else w.zero();
            reinterpret_cast<uint4*>(drow)[c] = encode_piece<N, PARTS>(p, w, g, ck, kb, part, bias, csum);
        }
        if (PARTS == 4 && p.is_weight) {
            const int32_t s = __reduce_add_sync(0xffffffffu, csum);
            if (lane == 0) {
                if (!LONG || wpr == 1) p.colsum[(r + i) * 2 + g] = s - (1 << (N - 1)) * 32 * p.blk_dst[g];
                else atomicAdd(sum, s);
            }
        }
    }
}

// LONG: rows shared by warps, or tiles off the 16-byte grid (the general form, whose run-time
// strides cost the others 3 to 13 %).
template <bool LONG>
__global__ void __launch_bounds__((kStreamWarps + 1) * 32, 4) expand_stream_kernel(const __grid_constant__ StreamParams sp) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full_bar[kStreamMaxStages], empty_bar[kStreamMaxStages];
    __shared__ uint32_t abort_s, none_s;
    __shared__ int32_t sums_s[kStreamMaxStages][kStreamWarps];    // code sums [row of the tile][group], wpr > 1
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t abort_flag = tc::smem_u32(&abort_s), base = tc::smem_u32(smem);
    if (threadIdx.x == 0) {
        for (int i = 0; i < sp.stages; ++i) {
            tc::mbar_init(tc::smem_u32(&full_bar[i]), 1);
            tc::mbar_init(tc::smem_u32(&empty_bar[i]), kStreamWarps);
        }
        tc::set_flag(abort_flag, 0);
        none_s = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (LONG && threadIdx.x < kStreamMaxStages * kStreamWarps) (&sums_s[0][0])[threadIdx.x] = 0;
    __syncthreads();
    tc::pdl_wait();      // launched with launch_pdl: the packed rows are written before this
    // (no early trigger: GEMM CTAs that move in as this kernel's leave cost the MLP block 14 us)
    const int wpr = LONG ? sp.wpr : 1, tr = kStreamWarps / wpr * sp.rpw;         // warps per row, rows per tile
    const int64_t tiles_a = (sp.op[0].rows + tr - 1) / tr;
    const int64_t tiles = tiles_a + (sp.op[1].rows + tr - 1) / tr;
    int b = 0;
    uint32_t ph = 0u;
    if (warp == kStreamWarps) {
        // ---- producer ----
        // writes out the code sums of weight tile t, in stage st, and clears them
        auto flush = [&](int64_t t, int st) {
            const ExpandParams& p = sp.op[1];
            const int64_t r = (t - tiles_a) * tr + (lane >> 1);
            const int g = lane & 1;
            if (t >= tiles_a && lane < 2 * tr && r < p.rows && p.kind[g] == 1 && p.blk_dst[g] > 0) {
                p.colsum[r * 2 + g] = sums_s[st][lane] - (1 << (p.bits[g] - 1)) * 32 * p.blk_dst[g];
                sums_s[st][lane] = 0;
            }
        };
        const int64_t behind = (int64_t)sp.stages * gridDim.x;
        bool ok = true;
        int64_t issued = 0;
        for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x, ++issued) {
            if (issued >= sp.stages) {
                ok = tc::wait_bounded_warp(tc::smem_u32(&empty_bar[b]), ph ^ 1u, abort_flag, kTimeoutNs, sp.err, kErrWait);
                if (!ok) break;
                if (LONG && wpr > 1) flush(t - behind, b);
            }
            const ExpandParams& p = sp.op[t < tiles_a ? 0 : 1];
            const int64_t r0 = (t < tiles_a ? t : t - tiles_a) * tr;
            const int nr = (int)(p.rows - r0 < tr ? p.rows - r0 : tr);
            // the tile keeps its global address modulo 16: one bulk copy of the aligned interior,
            // lanes 0..2 move the words before it, 4..6 those after it
            const uint8_t* src = p.src + r0 * p.src_row_bytes;
            const int shift = LONG ? (int)((uintptr_t)src & 15u) : 0, bytes = nr * (int)p.src_row_bytes;
            const int head = min((16 - shift) & 15, bytes), body = (bytes - head) & ~15, tail = bytes - head - body;
            const uint32_t dst = base + (uint32_t)(b * sp.stage_bytes + shift), bar = tc::smem_u32(&full_bar[b]);
            if (lane == 0 && body > 0) {
                asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(body)
                             : "memory");
                tc::bulk_load(dst + head, src + head, (uint32_t)body, bar);
            }
            const int at = lane < 4 ? 4 * lane : head + body + 4 * (lane - 4);
            if (lane < 4 ? 4 * lane < head : 4 * (lane - 4) < tail)
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + at), "r"(__ldg(reinterpret_cast<const uint32_t*>(src + at)))
                             : "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(bar);
            if (++b == sp.stages) {
                b = 0;
                ph ^= 1u;
            }
        }
        if (LONG && ok && wpr > 1) {
            // the code sums still in the ring
            for (int64_t i = issued > sp.stages ? issued - sp.stages : 0; i < issued && ok; ++i) {
                const int st = (int)(i % sp.stages);
                ok = tc::wait_bounded_warp(tc::smem_u32(&empty_bar[st]), (uint32_t)(i / sp.stages) & 1u, abort_flag,
                                           kTimeoutNs, sp.err, kErrWait);
                if (ok) flush(blockIdx.x + i * gridDim.x, st);
            }
        }
        // the copies in flight land before the CTA exits, also when it was abandoned
        if (lane == 0)
            for (int64_t i = issued > sp.stages ? issued - sp.stages : 0; i < issued; ++i)
                tc::wait_bounded(tc::smem_u32(&full_bar[i % sp.stages]), (uint32_t)(i / sp.stages) & 1u, tc::smem_u32(&none_s),
                                 kTimeoutNs, sp.err, kErrWait);
        return;
    }
    // ---- consumers: warp -> rows row0 .. row0 + rpw - 1 of a tile, pieces sub modulo wpr ----
    const int row0 = warp / wpr * sp.rpw, sub = warp % wpr;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        if (!tc::wait_bounded_warp(tc::smem_u32(&full_bar[b]), ph, abort_flag, kTimeoutNs, sp.err, kErrWait)) return;
        const ExpandParams& p = sp.op[t < tiles_a ? 0 : 1];
        const int64_t r0 = (t < tiles_a ? t : t - tiles_a) * tr, r = r0 + row0;
        const int nr = p.rows - r < sp.rpw ? (int)(p.rows - r) : sp.rpw;
        if (nr > 0) {
            uint32_t row = base + (uint32_t)(b * sp.stage_bytes) + (uint32_t)(row0 * (int)p.src_row_bytes);
            if (LONG) row += (uint32_t)(uintptr_t)(p.src + r0 * p.src_row_bytes) & 15u;
            asm volatile("" : "+r"(row)::"memory");        // keeps the row's loads behind the wait
#pragma unroll 1
            for (int g = 0; g < 2; ++g) {
                if (p.blk_dst[g] == 0) continue;
                const uint32_t src = row + (uint32_t)p.src_off[g];
                const int n = p.bits[g];
                int32_t* sum = &sums_s[b][2 * (warp / wpr) % kStreamWarps + g];
                auto group = [&](auto bits, auto parts) {
                    stream_group<decltype(bits)::value, decltype(parts)::value, LONG>(p, src, r, nr, g, lane, sub, wpr, sum);
                };
                using std::integral_constant;
                constexpr integral_constant<int, 1> c1{};
                constexpr integral_constant<int, 2> c2{};
                constexpr integral_constant<int, 4> c4{};
                if (p.kind[g] == 2) {
                    if (n == 1) group(c1, c1);
                    else group(c2, c1);
                } else if (p.kind[g] == 0) {
                    switch (n) {
                        case 1: group(c1, c2); break;
                        case 2: group(c2, c2); break;
                        case 3: group(integral_constant<int, 3>{}, c2); break;
                        default: group(c4, c2); break;
                    }
                } else {
                    switch (n) {
                        case 1: group(c1, c4); break;
                        case 2: group(c2, c4); break;
                        case 3: group(integral_constant<int, 3>{}, c4); break;
                        case 4: group(c4, c4); break;
                        case 5: group(integral_constant<int, 5>{}, c4); break;
                        case 6: group(integral_constant<int, 6>{}, c4); break;
                        case 7: group(integral_constant<int, 7>{}, c4); break;
                        default: group(integral_constant<int, 8>{}, c4); break;
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(tc::smem_u32(&empty_bar[b]));
        if (++b == sp.stages) {
            b = 0;
            ph ^= 1u;
        }
    }
}

// expand_stream_kernel for linear layers; false for convolutions, which gather their rows.
bool launch_stream(const ExpandParams& a, const ExpandParams& w, cudaStream_t st, cudaError_t* err) {
    if (a.conv) return false;
    const int64_t row = a.src_row_bytes > w.src_row_bytes ? a.src_row_bytes : w.src_row_bytes;
    // four CTAs per SM, or two where four rings of two stages do not fit (rows over 3.4 KB;
    // 8192 x 4096 x 4096 4/8 bits: two 101, three 99.7, four 99.4 us a call; 2/8 bits 81, 80, 79.6),
    // and then as few warps per row as two stages allow (two from 6.9 KB on, four, eight; the
    // longest row, 64 KB, has one CTA per SM)
    int per_sm = kStreamWarps * row * 2 + 256 <= (int64_t)kStreamSmemPerSm / 4 ? 4 : 2;
    int64_t wpr = 1;
    while (wpr < kStreamWarps && kStreamWarps / wpr * row * 2 + 288 > (int64_t)kStreamSmemPerSm / per_sm) wpr *= 2;
    if (kStreamWarps / wpr * row * 2 + 288 > (int64_t)kStreamSmemPerSm / per_sm) per_sm = 1;
    const int64_t smem_cta = (int64_t)kStreamSmemPerSm / per_sm;
    // short rows: several per warp and stage (about 12 KB), as long as every CTA gets two tiles
    // (16384 x 768 x 3072: 61 us a call, one row per warp 70)
    const int64_t cap = (int64_t)num_sms() * per_sm, all = a.rows + w.rows;
    int64_t rpw = 12 * 1024 / (kStreamWarps * row);
    if (rpw > all / (2 * cap * kStreamWarps)) rpw = all / (2 * cap * kStreamWarps);
    if (rpw > 4) rpw = 4;
    if (rpw < 1 || wpr > 1) rpw = 1;
    const int64_t tr = kStreamWarps / wpr * rpw;
    // (room to keep a tile's address modulo 16 where tiles do not start on that grid)
    const bool grid16 = ((uintptr_t)a.src | (uintptr_t)w.src | (uintptr_t)(tr * a.src_row_bytes) |
                         (uintptr_t)(tr * w.src_row_bytes)) % 16 == 0;
    const int64_t stage = (tr * row + (grid16 ? 0 : 16) + 127) / 128 * 128;
    const int64_t stages = smem_cta / stage;
    if (stages < 2) return false;
    StreamParams sp;
    sp.op[0] = a;
    sp.op[1] = w;
    sp.err = device_error_word();
    if (sp.err == nullptr) return false;
    sp.stages = (int32_t)(stages < kStreamMaxStages ? stages : kStreamMaxStages);
    sp.stage_bytes = (int32_t)stage;
    sp.rpw = (int32_t)rpw;
    sp.wpr = (int32_t)wpr;
    const int64_t tiles = (a.rows + tr - 1) / tr + (w.rows + tr - 1) / tr;
    const bool is_long = wpr > 1 || !grid16;
    const auto fn = is_long ? expand_stream_kernel<true> : expand_stream_kernel<false>;
    static bool attr_done[64][2] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return false;
    if (!attr_done[dev][is_long]) {
        *err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStreamSmemPerSm);
        if (*err == cudaSuccess) *err = prefer_max_shared((const void*)fn);
        if (*err != cudaSuccess) return true;
        attr_done[dev][is_long] = true;
    }
    *err = launch_pdl(fn, dim3((unsigned)(tiles < cap ? tiles : cap)), dim3((kStreamWarps + 1) * 32),
                      (size_t)(sp.stages * sp.stage_bytes), st, sp);
    return true;
}

// ---------------------------------------------------------------------------
// The persistent GEMM over expanded operands
// ---------------------------------------------------------------------------

// 8 consecutive outputs of row m from column nb (one 16-byte store when aligned).
__device__ __forceinline__ void store_out8(const SParams& p, int64_t m, int nb, const float (&y)[8]) {
    const bool vec = nb + 8 <= p.N && (p.N & 7) == 0;
    uint32_t wv[4];
    if (p.out_bf16) {
        __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.Y) + m * p.N;
        if (vec) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                __nv_bfloat162 h2 = __floats2bfloat162_rn(y[2 * e], y[2 * e + 1]);
                wv[e] = *reinterpret_cast<uint32_t*>(&h2);
            }
            *reinterpret_cast<uint4*>(dst + nb) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
        } else {
            for (int j = 0; j < 8; ++j)
                if (nb + j < p.N) dst[nb + j] = __float2bfloat16_rn(y[j]);
        }
    } else {
        __half* dst = reinterpret_cast<__half*>(p.Y) + m * p.N;
        if (vec) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                __half2 h2 = __floats2half2_rn(y[2 * e], y[2 * e + 1]);
                wv[e] = *reinterpret_cast<uint32_t*>(&h2);
            }
            *reinterpret_cast<uint4*>(dst + nb) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
        } else {
            for (int j = 0; j < 8; ++j)
                if (nb + j < p.N) dst[nb + j] = __float2half_rn(y[j]);
        }
    }
}

// The tile's accumulation jobs, in order: the group that needs exact
// segments (if any) first, then the other one; each segment is one job.
// Job k of the CTA accumulates into TMEM region k % 2 (256 columns), so the
// epilogue drains one region while the MMAs fill the other.
__device__ __forceinline__ int first_group(const SParams& p) { return p.seg_group == 1 ? 1 : 0; }

// Shared address of 8-column block c (0..3) of row r in a warp's 32 x 32 batch
// of staged outputs: 64-byte rows, swizzled so that 8 rows of a block, and the
// 4 blocks of 2 rows, lie on distinct banks.
__device__ __forceinline__ uint32_t batch_addr(uint32_t out_s, int c, int r) {
    return out_s + (uint32_t)r * 64u + ((((uint32_t)c) ^ (((uint32_t)r >> 1) & 3u)) << 4);
}

// Quantize-in-epilogue (Sec. 4.1, Conv2D + BatchNorm + Quantize fused): the
// next layer's packed codes of this lane's row from the fp16 outputs in the
// warp's staging tile (row `lane`, 128 columns from nc0, 64-column boxes of
// 128-byte-swizzled rows).  The columns are the next layer's packed
// positions, so each 32-column block is one packed block of its group (Sec. 3
// step 2 with the next layer's calibrated scale).  Kept out of the unrolled
// output loop, with run-time widths, so that the kernel's code stays small.
__device__ __noinline__ void next_layer_codes(const SParams& p, uint32_t out_s, int lane, int64_t m, int nc0) {
    constexpr int COLS = 128;
    const QConst kn0 = make_qconst(__ldg(p.s_next), p.next_bits[0]);
    const QConst kn1 = make_qconst(__ldg(p.s_next + 1), p.next_bits[1]);
#pragma unroll 1
    for (int b = 0; b < COLS / 32; ++b) {
        const int cb = nc0 + 32 * b;                       // first column of the block
        if (cb >= p.N) break;
        const int gn = cb >= p.next_pa0;
        const int jg = cb - (gn ? p.next_pa0 : 0);         // position within the group
        const QConst kn = gn ? kn1 : kn0;
        const int valid = (gn ? p.next_count[1] : p.next_count[0]) - jg;   // real channels in the block
        uint32_t o[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int cc = 4 * b + i;                      // 8-column chunk of the staging tile
            const uint32_t src = out_s + (uint32_t)(cc >> 3) * 4096u + (uint32_t)lane * 128u +
                                 ((((uint32_t)cc & 7u) ^ ((uint32_t)lane & 7u)) << 4);
            uint32_t h[4];
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(h[0]), "=r"(h[1]), "=r"(h[2]), "=r"(h[3])
                         : "r"(src)
                         : "memory");
            uint32_t u[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[e]));
                u[2 * e] = act_code_q<true>(f.x, kn.s, kn.r, kn.levels, kn.top);
                u[2 * e + 1] = act_code_q<true>(f.y, kn.s, kn.r, kn.levels, kn.top);
            }
            if (kn.mode != 1) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h[e]));
                    u[2 * e] = kn.mode == 0 ? 0u : act_code_q<false>(f.x, kn.s, kn.r, kn.levels, kn.top);
                    u[2 * e + 1] = kn.mode == 0 ? 0u : act_code_q<false>(f.y, kn.s, kn.r, kn.levels, kn.top);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (8 * i + q >= valid) u[q] = 0u;         // padding positions hold code 0
            o[2 * i] = u[0] | (u[1] << 8) | (u[2] << 16) | (u[3] << 24);
            o[2 * i + 1] = u[4] | (u[5] << 8) | (u[6] << 16) | (u[7] << 24);
        }
        const int nb = gn ? p.next_bits[1] : p.next_bits[0];
        store_block32_rt(nb, o, p.Ap_next + m * p.next_row_bytes + (gn ? p.next_off[1] : p.next_off[0]) +
                                    (jg >> 5) * 4 * nb);
    }
}

// ---------------------------------------------------------------------------
// Fragment epilogue
// ---------------------------------------------------------------------------
//
// What bounds it: next to the MMAs' operand traffic, shared-memory bandwidth
// and instruction issue.  With one accumulator row per lane (the GENERAL
// epilogue) every lane reads every column's constants, 16 bytes per output
// element from shared memory, and each output takes four int/float
// conversions, which issue at a sixteenth of the fp32 rate.  Two changes:
//   * the accumulators are read as MMA fragments (tcgen05.ld 16x256b): a lane
//     holds columns 8 c + 2 (lane % 4) + {0, 1} of rows lane / 4 + {0, 8, 16,
//     24}, so one pair of 16-byte constants serves eight outputs, and
//     stmatrix writes the 8 x 8 blocks to the staging tile;
//   * an accumulator of one exact piece is an integer below 2^24 held in
//     fp32: v * 2^18 (or 4, or 1) is that integer, and adding the centring
//     term (an integer with at most 24 significant bits, also exact) rounds
//     once, to the very value the conversion of the int32 sum gives.
// Only segmented groups, whose sums may pass 2^24, go through int32.

struct FragTile {
    uint32_t bar0, abort_flag;
    uint32_t tmem;             // the warp's TMEM lane quadrant and first column of region 0
    uint32_t out_s;            // staging tile (shared address)
    float4* colc;              // column constants (shared memory)
    int quad, lane;
    int cgrp;                  // column half of the tile
    int tile;                  // tiles of this CTA so far
    int64_t m0;                // first row of the warp's 32
    int nc0;                   // its first column
};

#define SONIQ_R8(r, o) \
    "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
#define SONIQ_RW8(r, o) \
    "+r"(r[o]), "+r"(r[o + 1]), "+r"(r[o + 2]), "+r"(r[o + 3]), "+r"(r[o + 4]), "+r"(r[o + 5]), "+r"(r[o + 6]), "+r"(r[o + 7])

// Issues the loads of NC 8-column blocks of the quadrant's lanes 0..15 (v[0 ..
// 4 NC - 1]) and 16..31 (v[8 ..], 4 NC of them).  v[4 j + {0, 1}]: row lane / 4,
// columns 8 j + 2 (lane % 4) + {0, 1}; v[4 j + {2, 3}]: row lane / 4 + 8.  The
// values are there after tmem_frag_wait on the same registers.
template <int NC>
__device__ __forceinline__ void tmem_frag_issue(uint32_t taddr, uint32_t (&v)[16]) {
    const uint32_t hi = taddr + (16u << 16);
    if constexpr (NC == 2) {
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];"
            : SONIQ_R8(v, 0), SONIQ_R8(v, 8)
            : "r"(taddr), "r"(hi));
    } else {
        static_assert(NC == 1, "1 or 2 blocks");
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%8];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {%4,%5,%6,%7}, [%9];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11])
            : "r"(taddr), "r"(hi));
        v[4] = v[5] = v[6] = v[7] = v[12] = v[13] = v[14] = v[15] = 0u;
    }
}

// Waits for this thread's TMEM loads; v's registers pass through, so that no use of them moves up.
__device__ __forceinline__ void tmem_frag_wait(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : SONIQ_RW8(v, 0), SONIQ_RW8(v, 8)::"memory");
}

// Calls f(block, values) for 8-column blocks C .. NCH - 1, whose first two are
// in (or on their way to) cur; the next two load while these are processed.
// f's values: {0, 1} row lane / 4, {2, 3} + 8, {4, 5} + 16, {6, 7} + 24.
template <int C, int NCH, typename F>
__device__ __forceinline__ void frag_step(uint32_t taddr, uint32_t (&cur)[16], F& f) {
    constexpr int N = NCH - C >= 2 ? 2 : 1;
    tmem_frag_wait(cur);
    uint32_t nxt[16];
    if constexpr (C + N < NCH) tmem_frag_issue<(NCH - C - N >= 2 ? 2 : 1)>(taddr + 8 * (C + N), nxt);
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const uint32_t v[8] = {cur[4 * j], cur[4 * j + 1], cur[4 * j + 2], cur[4 * j + 3],
                               cur[8 + 4 * j], cur[9 + 4 * j], cur[10 + 4 * j], cur[11 + 4 * j]};
        f(C + j, v);
    }
    if constexpr (C + N < NCH) frag_step<C + N, NCH>(taddr, nxt, f);
}

template <int NCH, typename F>
__device__ __forceinline__ void frag_blocks(uint32_t taddr, F&& f) {
    uint32_t first[16];
    tmem_frag_issue<(NCH >= 2 ? 2 : 1)>(taddr, first);
    frag_step<0, NCH>(taddr, first, f);
}

// Four 8 x 8 blocks of 16-bit values (rows 0..31 of the warp); lane l gives the address of row l.
__device__ __forceinline__ void stmatrix4(uint32_t addr, const uint32_t (&w)[4]) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3]));
}

__device__ __forceinline__ uint32_t pack_out(float lo, float hi, int bf16) {
    if (bf16) {
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&h);
    }
    __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// The warp's staged batch, columns cb .. cb + 8 nc - 1 of its 32 rows, to Y:
// 16-byte stores, 64 contiguous bytes per row, or 4- or 2-byte ones where the
// row pitch (N) is not a multiple of 8.  (TMA stores would share the TMA unit
// with the operand loads.)
__device__ __forceinline__ void batch_out(const SParams& p, const FragTile& t, int cb, int nc) {
    __syncwarp();
    const int ncol = min(8 * nc, p.N - cb);
    if ((p.N & 7) == 0) {
        const int c = t.lane & 3;
        uint4* dst = reinterpret_cast<uint4*>(static_cast<uint16_t*>(p.Y) + (t.m0 + (t.lane >> 2)) * p.N + cb + 8 * c);
        const int64_t rows = p.M - t.m0 - (t.lane >> 2);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint4 v;
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                         : "r"(batch_addr(t.out_s, c, (t.lane >> 2) + 8 * i)));
            if (8 * c < ncol && 8 * i < rows) dst[(int64_t)i * p.N] = v;       // 8 rows: N 16-byte vectors
        }
    } else if ((p.N & 1) == 0) {
        const int c = 2 * (t.lane & 15);
        for (int r = t.lane >> 4; r < 32 && t.m0 + r < p.M; r += 2) {
            uint32_t v;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(batch_addr(t.out_s, c >> 3, r) + 2u * (c & 7)));
            if (c < ncol) *reinterpret_cast<uint32_t*>(static_cast<uint16_t*>(p.Y) + (t.m0 + r) * p.N + cb + c) = v;
        }
    } else {
        const int c = t.lane;
        for (int r = 0; r < 32 && t.m0 + r < p.M; ++r) {
            uint16_t v;
            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(batch_addr(t.out_s, c >> 3, r) + 2u * (c & 7)));
            if (c < ncol) static_cast<uint16_t*>(p.Y)[(t.m0 + r) * p.N + cb + c] = v;
        }
    }
    __syncwarp();      // read before the next batch is staged
}

// Shared address of row r of 8-column block c of a warp's whole staged tile:
// 64-column boxes of 128-byte-swizzled rows (the TMA store map's layout).
__device__ __forceinline__ uint32_t staging_addr(uint32_t out_s, int c, int r) {
    return out_s + (uint32_t)(c >> 3) * 4096u + (uint32_t)r * 128u + ((((uint32_t)c & 7u) ^ ((uint32_t)r & 7u)) << 4);
}

// The warp's whole staged tile leaves by TMA stores; rows and columns beyond M
// and N are clipped.
template <int EPI_COLS>
__device__ __forceinline__ void staged_out(const SParams& p, const FragTile& t) {
    static_assert(EPI_COLS % 64 == 0, "whole boxes");
    fence_proxy_async_shared();
    __syncwarp();
    if (t.lane == 0) {
#pragma unroll
        for (int bx = 0; bx < EPI_COLS / 64; ++bx)
            tma_store_2d(&p.tma_y, t.nc0 + bx * 64, (int)t.m0, t.out_s + bx * 4096u);
        bulk_commit();
    }
}

// Low bytes of four words, in order.
__device__ __forceinline__ uint32_t low_bytes(uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3) {
    return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
}

// Sec. 3 step 2 on a pair of fp16 outputs under a calibrated scale (Markstein
// quotient, the top clip on the input, its last step saturated to [0, 1], rounding
// by adding 1.5 * 2^23: the codes are the low bytes of the results).
__device__ __forceinline__ void next_codes2(uint32_t h2, const QConst& k, uint32_t& c0, uint32_t& c1) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h2));
    const float2 x = make_float2(fmin_keep_nan(f.x, k.s), fmin_keep_nan(f.y, k.s));
    const float2 q0 = mul2(x, make_float2(k.r, k.r));
    const float2 e = fma2(q0, make_float2(-k.s, -k.s), x);
    const float2 q = make_float2(fma_sat(e.x, k.r, q0.x), fma_sat(e.y, k.r, q0.y));
    const float2 u = add2(mul2(q, make_float2(k.levels, k.levels)), 12582912.0f);
    c0 = __float_as_uint(u.x);
    c1 = __float_as_uint(u.y);
}

// The next layer's packed codes from the warp's code bytes: cw[4 j + i] holds,
// for 16-column block j and rows 8 i + lane / 4, the bytes of columns
// 16 j + 2 (lane % 4) + {0, 1} and 16 j + 8 + 2 (lane % 4) + {0, 1}.  They
// pass through the staging tile (128 bytes per row, swizzled); lane l then
// packs row l, one 32-column block of one group at a time.
template <int EPI_COLS>
__device__ __forceinline__ void next_pack(const SParams& p, const FragTile& t, const uint32_t (&cw)[EPI_COLS / 4]) {
    static_assert(EPI_COLS == 128, "128-byte rows");
#pragma unroll
    for (int j = 0; j < EPI_COLS / 16; ++j) {
        const uint32_t w[4] = {cw[4 * j], cw[4 * j + 1], cw[4 * j + 2], cw[4 * j + 3]};
        stmatrix4(staging_addr(t.out_s, j, t.lane), w);
    }
    __syncwarp();
    const int64_t m = t.m0 + t.lane;
    if (m >= p.M) return;
    uint8_t* dst = p.Ap_next + m * p.next_row_bytes;
#pragma unroll 1
    for (int b = 0; b < EPI_COLS / 32; ++b) {
        const int cb = t.nc0 + 32 * b;                     // first column of the block
        if (cb >= p.N) break;
        const int gn = cb >= p.next_pa0;
        const int jg = cb - (gn ? p.next_pa0 : 0);         // position within the group
        uint32_t o[8];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t w[4];
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                         : "r"(staging_addr(t.out_s, 2 * b + i, t.lane))
                         : "memory");
            // word q: columns 2q, 2q + 1 of the first eight (low half) and of the second eight
            o[4 * i] = __byte_perm(w[0], w[1], 0x5410);
            o[4 * i + 1] = __byte_perm(w[2], w[3], 0x5410);
            o[4 * i + 2] = __byte_perm(w[0], w[1], 0x7632);
            o[4 * i + 3] = __byte_perm(w[2], w[3], 0x7632);
        }
        const int valid = (gn ? p.next_count[1] : p.next_count[0]) - jg;   // real channels in the block
        if (valid < 32) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int v = valid - 4 * q;               // padding positions hold code 0
                o[q] &= v >= 4 ? 0xFFFFFFFFu : (v <= 0 ? 0u : (1u << (8 * v)) - 1u);
            }
        }
        const int nb = gn ? p.next_bits[1] : p.next_bits[0];
        store_block32_n(nb, o, dst + (gn ? p.next_off[1] : p.next_off[0]) + (jg >> 5) * 4 * nb);
    }
}

// How a layer's tiles end: group gl completes with the tile's last job; group
// gf (the first job's, or an absent one) is in registers by then.
template <int EPI>
struct ColPlan {
    int gA, nA, njobs;         // the first jobs' group, its jobs, all jobs of a tile
    int gf, gl;
    bool both, same;           // two groups; SEG: earlier segments are of group gl itself
    float invf, invl, scf, scl;
    int centf, centl;          // centring of group f / l (0: none)
    float saf, sal;            // per-tensor activation scales (1: per row)
    __device__ __forceinline__ explicit ColPlan(const SParams& p) {
        gA = kEpiSegments<EPI> ? first_group(p) : 0;   // in segments only group gA may be
        const int gB = 1 - gA;
        nA = p.g[gA].stages > 0 ? p.g[gA].n_seg : 0;
        const int nB = p.g[gB].stages > 0 ? p.g[gB].n_seg : 0;
        njobs = nA + nB;
        gl = nB > 0 ? gB : gA;
        gf = 1 - gl;
        both = nA > 0 && nB > 0;
        same = kEpiSegments<EPI> && !both;
        invf = p.g[gf].inv_levels;
        invl = p.g[gl].inv_levels;
        scf = p.g[gf].acc_scale;
        scl = p.g[gl].acc_scale;
        centf = both ? p.g[gf].center : 0;
        centl = p.g[gl].center;
        saf = p.s_a_per_row ? 1.0f : __ldg(p.s_a + gf);
        sal = p.s_a_per_row ? 1.0f : __ldg(p.s_a + gl);
    }
};

// A tile's column constants {scale f, scale l, centring f, centring l}
// (per-tensor: s_a included), 32 bytes per column pair: {scale f x 2, scale l
// x 2}, {centring f x 2, centring l x 2}.  The four warps of a column half
// each prepare a quarter of them: the global loads are issued before the
// previous tile's last job, the stores follow it, and the half's barrier (one
// per buffer) says that all four have arrived.
struct ColLoad {
    float2 sw;
    int cf, cl;
    template <int EPI>
    __device__ __forceinline__ void load(const SParams& p, const ColPlan<EPI>& cp, const FragTile& t, int epi_cols) {
        const int c = t.quad * (epi_cols / 4) + t.lane;
        const int n = t.nc0 + c < p.N ? t.nc0 + c : p.N - 1;
        // two scalar loads: s_w is 4-byte aligned, no more
        sw = make_float2(__ldg(p.s_w + (int64_t)n * 2), __ldg(p.s_w + (int64_t)n * 2 + 1));
        cf = cp.centf ? __ldg(p.colsum + (int64_t)n * 2 + cp.gf) : 0;
        cl = cp.centl ? __ldg(p.colsum + (int64_t)n * 2 + cp.gl) : 0;
    }
    // into the buffer of tile number t.tile
    template <typename C, int EPI>
    __device__ __forceinline__ void store(const ColPlan<EPI>& cp, const FragTile& t) {
        const int buf = t.tile & 1;
        if (t.lane < C::EPI_COLS / 4) {
            const int c = t.quad * (C::EPI_COLS / 4) + t.lane;
            float* d = reinterpret_cast<float*>(t.colc) + buf * (C::COLS_BYTES / 4) + (c >> 1) * 8 + (c & 1);
            d[0] = __fmul_rn(cp.saf, (cp.gf ? sw.y : sw.x) * cp.invf);
            d[2] = __fmul_rn(cp.sal, (cp.gl ? sw.y : sw.x) * cp.invl);
            // int32 where the group's sum is one, else fp32 (exact)
            const int f = cp.centf * cf, l = cp.centl * cl;
            d[4] = kEpiSegments<EPI> ? __int_as_float(f) : (float)f;
            d[6] = cp.same ? __int_as_float(l) : (float)l;
        }
        __syncwarp();
        if (t.lane == 0) mbar_arrive(t.bar0 + 8u * (uint32_t)(C::BAR_COLS + 2 * t.cgrp + buf));
    }
};

// One tile of an epilogue warp: waits for the tile's jobs, drains them and
// writes the outputs (NEXT: also the next layer's codes); prepares tile nxt's
// column constants (nxt.nc0 < 0: there is none).  release(r) hands TMEM region
// r back.  False after a wait ran out.
template <int EPI, bool ROWS, int BNT, bool PAIR, int OUT, typename Release>
__device__ __forceinline__ bool frag_tile(const SParams& p, const ColPlan<EPI>& cp, const FragTile& t, FragTile& nxt,
                                          ColLoad& cl, uint32_t& job, Release&& release) {
    using C = Cfg<BNT, PAIR, OUT>;
    constexpr int EPI_COLS = C::EPI_COLS, NCH = EPI_COLS / 8;
    constexpr bool SEG = kEpiSegments<EPI>, NEXT = kEpiNext<EPI>;
    const int lane = t.lane;
    auto wait = [&](int b, uint32_t ph) {
        return __all_sync(0xffffffffu, wait_bounded(t.bar0 + 8u * (uint32_t)b, ph, t.abort_flag, kTimeoutNs, p.err,
                                                    kErrWait)) != 0;
    };
    // activation scales of this lane's four rows, groups f and l
    float2 saf[4], sal[4];
    if constexpr (ROWS) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t m = t.m0 + 8 * r + (lane >> 2);
            float f = 1.0f, l = 1.0f;
            if (p.s_a_per_row) {
                f = m < p.M ? __ldg(p.s_a + m * 2 + cp.gf) : 0.0f;
                l = m < p.M ? __ldg(p.s_a + m * 2 + cp.gl) : 0.0f;
            }
            saf[r] = make_float2(f, f);
            sal[r] = make_float2(l, l);
        }
    }

    // ---- earlier jobs: the whole first group, or segments ----
    uint32_t part[NCH * 8];                          // accumulators as they are, or int32 sums (SEG)
#pragma unroll
    for (int i = 0; i < NCH * 8; ++i) part[i] = 0u;
#pragma unroll 1
    for (int jj = 0; jj < cp.njobs - 1; ++jj, ++job) {
        const uint32_t r = job & 1u, use = job >> 1;
        if (!wait(C::BAR_REG_FULL + (int)r, use & 1u)) return false;
        tc_fence_after();
        const float sc = p.g[jj < cp.nA ? cp.gA : 1 - cp.gA].acc_scale;
        frag_blocks<NCH>(t.tmem + r * REGION, [&](int c, const uint32_t (&v)[8]) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if constexpr (SEG) part[8 * c + e] += (uint32_t)__float2int_rn(__fmul_rn(__uint_as_float(v[e]), sc));
                else part[8 * c + e] = v[e];
            }
        });
        tc_fence_before();
        __syncwarp();
        if (lane == 0) release(r);
    }

    // ---- the final job ----
    if (nxt.nc0 >= 0) cl.load(p, cp, nxt, EPI_COLS);
    const int buf = t.tile & 1;
    if (!wait(C::BAR_COLS + 2 * t.cgrp + buf, (uint32_t)(t.tile >> 1) & 1u)) return false;
    const uint32_t r = job & 1u, use = job >> 1;
    ++job;
    if (!wait(C::BAR_REG_FULL + (int)r, use & 1u)) return false;
    tc_fence_after();
    QConst kn0, kn1;
    bool codes_here = false;
    if constexpr (NEXT) {
        kn0 = make_qconst(__ldg(p.s_next), p.next_bits[0]);
        kn1 = make_qconst(__ldg(p.s_next + 1), p.next_bits[1]);
        // scales outside the Markstein range: from the staged outputs, below
        codes_here = kn0.mode == 1 && kn1.mode == 1;
    }
    const bool stage_y = !NEXT || p.write_y || !codes_here;
    if constexpr (OUT == OUT_TMA) {
        // the previous tile's store must have read the staging tile
        if (lane == 0) bulk_wait_read0();
        __syncwarp();
    }
    const float4* kc = t.colc + buf * (C::COLS_BYTES / 16) + 2 * (lane & 3);
    const float2 scf = make_float2(cp.scf, cp.scf), scl = make_float2(cp.scl, cp.scl);
    uint32_t cw[NEXT ? EPI_COLS / 4 : 1];
    uint32_t cprev[NEXT ? 8 : 1];
    frag_blocks<NCH>(t.tmem + r * REGION, [&](int c, const uint32_t (&v)[8]) {
        const float4 ks = kc[8 * c], ct = kc[8 * c + 1];     // scales, centrings of the lane's two columns
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {                          // row lane / 4 + 8 i
            float2 kf = make_float2(ks.x, ks.y), kl = make_float2(ks.z, ks.w);
            if constexpr (ROWS) {
                kf = mul2(saf[i], kf);
                kl = mul2(sal[i], kl);
            }
            const float2 vl = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
            const uint32_t p0 = part[8 * c + 2 * i], p1 = part[8 * c + 2 * i + 1];
            float2 y;
            if constexpr (SEG) {
                float2 xl, xf;
                if (cp.same) {
                    const int x0 = (int)p0 + __float2int_rn(__fmul_rn(vl.x, cp.scl)) + __float_as_int(ct.z);
                    const int x1 = (int)p1 + __float2int_rn(__fmul_rn(vl.y, cp.scl)) + __float_as_int(ct.w);
                    xl = make_float2((float)x0, (float)x1);
                    xf = make_float2(0.0f, 0.0f);
                } else {
                    xl = fma2(vl, scl, make_float2(ct.z, ct.w));
                    xf = make_float2((float)((int)p0 + __float_as_int(ct.x)), (float)((int)p1 + __float_as_int(ct.y)));
                }
                // group 0's product is rounded first
                y = cp.gf == 0 ? fma2(kl, xl, mul2(kf, xf)) : fma2(kf, xf, mul2(kl, xl));
            } else {
                const float2 vf = make_float2(__uint_as_float(p0), __uint_as_float(p1));
                const float2 xl = fma2(vl, scl, make_float2(ct.z, ct.w));
                const float2 xf = fma2(vf, scf, make_float2(ct.x, ct.y));
                y = fma2(kl, xl, mul2(kf, xf));
            }
            w[i] = pack_out(y.x, y.y, NEXT ? 0 : p.out_bf16);
        }
        if (stage_y) stmatrix4(OUT == OUT_BATCH ? batch_addr(t.out_s, c & 3, lane) : staging_addr(t.out_s, c, lane), w);
        if constexpr (NEXT) {
            // a 32-column block has one group, so this test is warp-uniform
            const bool g1 = t.nc0 + 8 * c >= p.next_pa0;
            QConst k;
            k.s = g1 ? kn1.s : kn0.s;
            k.r = g1 ? kn1.r : kn0.r;
            k.levels = g1 ? kn1.levels : kn0.levels;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t c0, c1;
                next_codes2(w[i], k, c0, c1);
                if (c & 1) cw[4 * (c >> 1) + i] = low_bytes(cprev[2 * i], cprev[2 * i + 1], c0, c1);
                cprev[2 * i] = c0;
                cprev[2 * i + 1] = c1;
            }
        }
        if constexpr (OUT == OUT_BATCH)
            if ((c & 3) == 3 || c == NCH - 1) batch_out(p, t, t.nc0 + 32 * (c >> 2), (c & 3) + 1);
    });
    tc_fence_before();
    __syncwarp();
    if (lane == 0) release(r);
    if constexpr (OUT == OUT_TMA)
        if (!NEXT || p.write_y) staged_out<EPI_COLS>(p, t);
    if (nxt.nc0 >= 0) {
        nxt.tile = t.tile + 1;
        cl.store<C>(cp, nxt);
    }
    if constexpr (NEXT) {
        if (codes_here) {
            if (p.write_y) {
                if (lane == 0) bulk_wait_read0();    // the outputs' store has read the staging tile
                __syncwarp();
            }
            next_pack<EPI_COLS>(p, t, cw);
        } else {
            __syncwarp();
            if (t.m0 + lane < p.M) next_layer_codes(p, t.out_s, lane, t.m0 + lane, t.nc0);
        }
        __syncwarp();
    }
    return true;
}

// Scale runs along K, one tile of an epilogue warp: every job is one run b of
// one group g, whose exact integer sum is added in fp32 with its own scale,
// y += (s_a(g, b) s_w(n, g, b) / (La Lw)) * Acc(g, b).  A job's scales are
// loaded while the previous job is drained.  DBG: acc_dbg receives [2][nb][M][N]
// (a run-time test per element, not taken, made a job's drain 2000 cycles instead
// of 320).  False after a wait ran out.
template <bool DBG, int BNT, bool PAIR, typename Release>
__device__ __forceinline__ bool runs_tile(const SParams& p, const FragTile& t, uint32_t& job, Release&& release) {
    using C = Cfg<BNT, PAIR, OUT_BATCH>;
    constexpr int EPI_COLS = C::EPI_COLS, NCH = EPI_COLS / 8, NK = EPI_COLS / 32;
    const int lane = t.lane;
    const int n0 = p.g[0].stages > 0 ? p.g[0].n_seg : 0, n1 = p.g[1].stages > 0 ? p.g[1].n_seg : 0;
    float* kcol = reinterpret_cast<float*>(t.colc);
    // scales of run jj: of the columns lane + 32 h, and of this lane's rows
    float kw[NK], sa[4];
    auto load_scales = [&](int jj) {
        const int g = jj < n0 ? 0 : 1, b = g ? jj - n0 : jj;
#pragma unroll
        for (int h = 0; h < NK; ++h) {
            const int n = t.nc0 + lane + 32 * h < p.N ? t.nc0 + lane + 32 * h : p.N - 1;
            kw[h] = __ldg(p.s_w + ((int64_t)n * 2 + g) * p.nb + b);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int64_t m = t.m0 + 8 * r + (lane >> 2);
            sa[r] = m < p.M ? __ldg(p.s_a + ((p.s_a_per_row ? m : 0) * 2 + g) * p.nb + b) : 0.0f;
        }
    };
    float y[NCH * 8];
#pragma unroll
    for (int i = 0; i < NCH * 8; ++i) y[i] = 0.0f;
    if (n0 + n1 > 0) load_scales(0);
#pragma unroll 1
    for (int jj = 0; jj < n0 + n1; ++jj, ++job) {
        const int g = jj < n0 ? 0 : 1, b = g ? jj - n0 : jj;
        const float sc = p.g[g].acc_scale, inv = p.g[g].inv_levels;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < NK; ++h)
            kcol[lane + 32 * h] = __fmul_rn(kw[h], inv);
        __syncwarp();
        const float s[4] = {sa[0], sa[1], sa[2], sa[3]};
        if (jj + 1 < n0 + n1) load_scales(jj + 1);
        const uint32_t r = job & 1u, use = job >> 1;
        if (!__all_sync(0xffffffffu, wait_bounded(t.bar0 + 8u * (C::BAR_REG_FULL + r), use & 1u, t.abort_flag,
                                                  kTimeoutNs, p.err, kErrWait)))
            return false;
        tc_fence_after();
        frag_blocks<NCH>(t.tmem + r * REGION, [&](int c, const uint32_t (&v)[8]) {
            const float2 kk = *reinterpret_cast<const float2*>(kcol + 8 * c + 2 * (lane & 3));
            const float k[2] = {kk.x, kk.y};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float x = __fmul_rn(__uint_as_float(v[e]), sc);       // the exact integer sum
                y[8 * c + e] = __fmaf_rn(__fmul_rn(s[e >> 1], k[e & 1]), x, y[8 * c + e]);
                if constexpr (DBG) {
                    const int64_t m = t.m0 + 8 * (e >> 1) + (lane >> 2);
                    const int n = t.nc0 + 8 * c + 2 * (lane & 3) + (e & 1);
                    if (m < p.M && n < p.N) p.acc_dbg[(((int64_t)g * p.nb + b) * p.M + m) * p.N + n] = __float2int_rn(x);
                }
            }
        });
        tc_fence_before();
        __syncwarp();
        if (lane == 0) release(r);
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = pack_out(y[8 * c + 2 * i], y[8 * c + 2 * i + 1], p.out_bf16);
        stmatrix4(batch_addr(t.out_s, c & 3, lane), w);
        if ((c & 3) == 3) batch_out(p, t, t.nc0 + 32 * (c >> 2), 4);
    }
    return true;
}

template <int EPI, bool ROWS, int BNT, bool PAIR, int OUT>
__global__ void __launch_bounds__(NUM_THREADS, 1) staged_mma_kernel(const __grid_constant__ SParams p) {
    // the tile width and what follows from it (BNT = 240: layouts with E2M1 groups,
    // whose block scale factors sit in the 16 TMEM columns past each region's tile)
    // PAIR: 2-SM MMAs.  CTAs run in clusters of two on a 256 x 256 tile: each
    // stages its own 128 A rows and its half of the B columns (32 KB per
    // K-stage instead of 48), the even-rank CTA issues M = 256 MMAs that read
    // both CTAs' stages, and each CTA's TMEM receives its own 128 rows.  Both
    // CTAs' operand bytes count on the issuing CTA's full barriers; its MMA
    // commits arrive on both CTAs' empty and region-full barriers; both CTAs'
    // epilogue warps arrive on its region-empty barriers.
    static_assert(!PAIR || (BNT / 2) % 8 == 0, "pairs split B boxes into halves of whole 8-row swizzle atoms");
    using C = Cfg<BNT, PAIR, OUT>;
    constexpr int BN = BNT;
    constexpr int STAGE_BYTES = C::STAGE_BYTES, STAGES = C::STAGES, EPI_COLS = C::EPI_COLS;
    constexpr int COLS_BYTES = C::COLS_BYTES, OUT_PER_WARP = C::OUT_PER_WARP;
    static_assert((EPI >= EPI_GENERAL) == (OUT == OUT_GENERAL) && (!kEpiNext<EPI> || OUT == OUT_TMA), "epilogue and outputs");
    constexpr int BAR_FULL = C::BAR_FULL, BAR_EMPTY = C::BAR_EMPTY, BAR_REG_FULL = C::BAR_REG_FULL,
                  BAR_REG_EMPTY = C::BAR_REG_EMPTY, BAR_TEARDOWN = C::BAR_TEARDOWN;
    constexpr int SMEM_OUT = C::SMEM_OUT, SMEM_COLS = C::SMEM_COLS, SMEM_BAR = C::SMEM_BAR, SMEM_MISC = C::SMEM_MISC;
    constexpr bool GENERAL = EPI == EPI_GENERAL || EPI == EPI_GENERAL_NEXT;
    constexpr bool F4 = BNT == BN_F4;    // layouts with E2M1 groups
    constexpr uint32_t IDESC2 = idesc(2 * BM, BN);
    constexpr uint32_t IDESC2_F4 = idesc_mxf4(2 * BM, BN);
    constexpr uint32_t IDESC = idesc(BM, BN);
    constexpr uint32_t IDESC_F4 = idesc_mxf4(BM, BN);
    constexpr bool BOX8 = EPI_COLS % 64 != 0;     // outputs leave in 8-column boxes
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(smem + SMEM_BAR);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + SMEM_MISC);
    const uint32_t abort_flag = smem_u32(smem + SMEM_MISC + 4);
    const uint32_t no_abort = smem_u32(smem + SMEM_MISC + 8);   // stays 0: waits that must run to completion
    const int g_first = first_group(p);
    if constexpr (PAIR) {
        // the pair instantiation works with cluster rank 1: outside a cluster
        // of two it reports the launch as invalid and does nothing
        if (cluster_size() != 2u) {
            if (threadIdx.x == 0) atomicOr(p.err, kErrWait);
            return;
        }
    }
    // the tiles this CTA walks: unit u of first_u, first_u + step_u, ... < n_units
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    const bool issuer = rank == 0u;                   // the CTA that issues the (2-SM) MMAs
    const int first_u = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int step_u = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
    const int n_units = PAIR ? p.pair_tiles : p.total_tiles;
    const int mp = (p.m_tiles + 1) >> 1;
    auto tile_m = [&](int u) { return PAIR ? 2 * (u % mp) + (int)rank : u % p.m_tiles; };
    auto tile_n = [&](int u) { return PAIR ? u / mp : u / p.m_tiles; };

    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) {
            mbar_init(bar(BAR_FULL + i), 1);
            mbar_init(bar(BAR_EMPTY + i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(BAR_REG_FULL + i), 1);
            mbar_init(bar(BAR_REG_EMPTY + i), PAIR ? 2 * NUM_EPI_WARPS : NUM_EPI_WARPS);
        }
        mbar_init(bar(BAR_TEARDOWN), 1);
        for (int i = 0; i < 4; ++i) mbar_init(bar(C::BAR_COLS + i), NUM_EPI_WARPS / 2);
        set_flag(abort_flag, 0);
        set_flag(no_abort, 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == WARP_MMA) {
        if constexpr (PAIR) {
            // one warp of each CTA of the pair allocates, collectively
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(tmem_slot)),
                         "r"(512)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(tmem_slot)),
                         "r"(512)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if constexpr (F4) {
        // the E2M1 block scale factors: UE8M0 2^0 in every byte of each region's
        // spare columns (one epilogue warp per TMEM lane quadrant)
        if (warp >= WARP_EPI && warp < WARP_EPI + 4) {
            const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
            tmem_st16(tmem_base + lanes + (uint32_t)BN_F4, 0x7F7F7F7Fu);
            tmem_st16(tmem_base + lanes + (uint32_t)(REGION + BN_F4), 0x7F7F7F7Fu);
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    // both CTAs' barriers (and scale factors) are in place before the peer's
    // loads, arrivals or MMAs reach them
    if constexpr (PAIR) cluster_sync();
    // launched with launch_pdl: the expanded operands and weight sums are
    // written before this (the prologue above touches no global memory)
    pdl_wait();

    // The launch gives every thread 168 registers; the epilogue's 128 partial
    // sums and loads in flight need more (168 spilled 40 of them), so the first
    // warpgroup hands its share over: 128 x 40 + 256 x 232 = 384 x 168.
    if (warp < WARP_EPI) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == WARP_TMA) {
            // -------------------------------------------------------- producer
            const bool leader = elect_one();
            uint32_t s = 0, slot = 0, ph = 0;
            bool ok = true;
            for (int u = first_u; u < n_units && ok; u += step_u) {
                const int m0 = tile_m(u) * BM, n0 = tile_n(u) * BN;
#pragma unroll 1
                for (int gi = 0; gi < 2 && ok; ++gi) {
                    const int g = gi == 0 ? g_first : 1 - g_first;
                    const int ns = p.g[g].stages, x0 = p.g[g].x0;
#pragma unroll 1
                    for (int i = 0; i < ns; ++i, ++s) {
                        if (!wait_bounded_warp(bar(BAR_EMPTY + slot), ph ^ 1u, abort_flag, kTimeoutNs, p.err,
                                               kErrWait)) {
                            ok = false;
                            break;
                        }
                        const uint32_t dst = sbase + slot * STAGE_BYTES;
                        if (p.drop_first && s == 0) {
                            // the MMA's wait for this stage runs out
                        } else if (leader) {
                            if constexpr (PAIR) {
                                // this CTA's A rows and B half; both CTAs' bytes complete on the
                                // issuing CTA's full barrier
                                const uint32_t fb = mapa_shared(bar(BAR_FULL + slot), 0u);
                                if (issuer) mbar_arrive_expect_tx(bar(BAR_FULL + slot), 2 * STAGE_BYTES);
                                tma_load_2d_pair(dst, &p.tma_a, x0 + i * KSTAGE, m0, fb);
                                tma_load_2d_pair(dst + A_BYTES, &p.tma_b, x0 + i * KSTAGE, n0 + (int)rank * (BN / 2),
                                                 fb);
                            } else {
                                mbar_arrive_expect_tx(bar(BAR_FULL + slot), STAGE_BYTES);
                                tma_load_2d(dst, &p.tma_a, x0 + i * KSTAGE, m0, bar(BAR_FULL + slot));
                                tma_load_2d(dst + A_BYTES, &p.tma_b, x0 + i * KSTAGE, n0, bar(BAR_FULL + slot));
                            }
                        }
                        __syncwarp();
                        if (++slot == (uint32_t)STAGES) {
                            slot = 0;
                            ph ^= 1u;
                        }
                    }
                }
            }
            // loads still in flight must land before the CTA's shared memory is released
            // (a pair's loads all complete on the issuing CTA's barriers; the other CTA
            // stays until the pair's final cluster barrier)
            if (!PAIR || issuer)
                for (uint32_t q = s > (uint32_t)STAGES ? s - STAGES : 0u; q < s; ++q)
                    if (!(p.drop_first && q == 0))
                        wait_bounded(bar(BAR_FULL + q % STAGES), (q / STAGES) & 1u, no_abort, kTimeoutNs, p.err,
                                     kErrWait);
        } else if (warp == WARP_MMA && issuer) {
            // -------------------------------------------------------------- MMA
            const bool leader = elect_one();
            uint32_t slot = 0, ph = 0, job = 0;
            bool ok = true;
            const uint64_t a_desc0 = sw128_desc(sbase);
            for (int u = first_u; u < n_units && ok; u += step_u) {
#pragma unroll 1
                for (int gi = 0; gi < 2 && ok; ++gi) {
                    const int g = gi == 0 ? g_first : 1 - g_first;
                    const int ns = p.g[g].stages;
                    const bool f8 = p.g[g].kind == 0, f4 = p.g[g].kind == 2;
                    const int per_job = p.g[g].n_seg > 1 ? p.g[g].seg_stages : ns;
#pragma unroll 1
                    for (int i = 0; i < ns && ok; ++job) {
                        const uint32_t r = job & 1u, use = job >> 1;
                        if (!wait_bounded_warp(bar(BAR_REG_EMPTY + r), (use & 1u) ^ 1u, abort_flag, kTimeoutNs, p.err,
                                               kErrWait)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t d = tmem_base + r * REGION;
                        const int jn = per_job < ns - i ? per_job : ns - i;
#pragma unroll 1
                        for (int q = 0; q < jn; ++q, ++i) {
                            if (!wait_bounded_warp(bar(BAR_FULL + slot), ph, abort_flag, kTimeoutNs, p.err, kErrWait)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            // descriptors of this stage; +32 bytes of K is +2 in the start-address field
                            const uint64_t ad = a_desc0 + (uint64_t)((slot * STAGE_BYTES) >> 4);
                            const uint64_t bd = ad + (uint64_t)(A_BYTES >> 4);
                            const uint32_t sf = d + (uint32_t)BN_F4;   // E2M1: this region's unit block scales
                            if (leader) {
                                // (one unrolled run of MMAs per operand kind: the kind's branch
                                // inside the run cost the headline call 12 us)
                                auto run = [&](auto&& mma) {
#pragma unroll
                                    for (int k = 0; k < KSTAGE / 32; ++k)
                                        mma(ad + 2 * k, bd + 2 * k, (q == 0 && k == 0) ? 0u : 1u);
                                };
                                if (F4 && f4) {
                                    run([&](uint64_t x, uint64_t y, uint32_t acc) {
                                        if constexpr (PAIR) mma2_f4(d, x, y, IDESC2_F4, sf, sf + 8u, acc);
                                        else mma_f4(d, x, y, IDESC_F4, sf, sf + 8u, acc);
                                    });
                                } else if (f8) {
                                    run([&](uint64_t x, uint64_t y, uint32_t acc) {
                                        if constexpr (PAIR) mma2_f8<IDESC2>(d, x, y, acc);
                                        else mma_f8<IDESC>(d, x, y, acc);
                                    });
                                } else {
                                    run([&](uint64_t x, uint64_t y, uint32_t acc) {
                                        if constexpr (PAIR) mma2_f16<IDESC2>(d, x, y, acc);
                                        else mma_f16<IDESC>(d, x, y, acc);
                                    });
                                }
                                // the stage's slot is free again (in both CTAs)
                                if constexpr (PAIR) mma2_commit_mc(bar(BAR_EMPTY + slot), (uint16_t)0x3);
                                else mma_commit(bar(BAR_EMPTY + slot));
                            }
                            __syncwarp();
                            if (++slot == (uint32_t)STAGES) {
                                slot = 0;
                                ph ^= 1u;
                            }
                        }
                        if (ok && leader) {
                            if constexpr (PAIR) mma2_commit_mc(bar(BAR_REG_FULL + r), (uint16_t)0x3);
                            else mma_commit(bar(BAR_REG_FULL + r));
                        }
                    }
                }
            }
            // every issued MMA completes before TMEM and shared memory are released
            if (leader) {
                if constexpr (PAIR) mma2_commit(bar(BAR_TEARDOWN));
                else mma_commit(bar(BAR_TEARDOWN));
            }
            __syncwarp();
            wait_bounded(bar(BAR_TEARDOWN), 0u, no_abort, kTimeoutNs, p.err, kErrWait);
        }
    } else {
        // ------------------------------------------------------------- epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
        // Warp w reads TMEM lane quadrant w % 4 (rows 32*(w%4) .. +31 of the
        // tile) and the EPI_COLS columns from cgrp * EPI_COLS, cgrp = (w - 4) / 4.
        const int ew = warp - WARP_EPI;
        const int quad = warp & 3;
        const int cgrp = ew >> 2;
        const int row = quad * 32 + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(cgrp * EPI_COLS);
        // column constants (GENERAL: this warp's copy, per column {s_w0 * inv_levels0,
        // s_w1 * inv_levels1, center0 * C0, center1 * C1}; the others: FragTile::colc)
        float4* colc = reinterpret_cast<float4*>(smem + SMEM_COLS + ew * COLS_BYTES);
        const uint32_t out_s = sbase + (uint32_t)(SMEM_OUT + ew * OUT_PER_WARP);   // 1024-aligned
        // a drained TMEM region goes back to the CTA that issues the MMAs
        auto release_region = [&](uint32_t r) {
            if (PAIR && !issuer) mbar_arrive_cluster(mapa_shared(bar(BAR_REG_EMPTY + (int)r), 0u));
            else mbar_arrive(bar(BAR_REG_EMPTY + (int)r));
        };
        uint32_t job = 0;
        bool ok = true;
        if constexpr (!GENERAL) {
            FragTile ft;
            ft.bar0 = bar0;
            ft.abort_flag = abort_flag;
            ft.tmem = lane_base;
            ft.out_s = out_s;
            ft.quad = quad;
            ft.lane = lane;
            ft.cgrp = cgrp;
            ft.tile = 0;
            // RUNS: a buffer per warp; else two per column half, in turn
            ft.colc = reinterpret_cast<float4*>(smem + SMEM_COLS + (EPI == EPI_RUNS ? ew : 2 * cgrp) * COLS_BYTES);
            auto place = [&](int u) {
                ft.m0 = (int64_t)tile_m(u) * BM + quad * 32;
                ft.nc0 = tile_n(u) * BN + cgrp * EPI_COLS;
            };
            if constexpr (EPI == EPI_RUNS) {
                for (int u = first_u; u < n_units && ok; u += step_u) {
                    place(u);
                    ok = runs_tile<ROWS, BNT, PAIR>(p, ft, job, release_region);
                }
            } else if (first_u < n_units) {
                const ColPlan<EPI> cp(p);
                ColLoad cl;
                place(first_u);
                cl.load(p, cp, ft, EPI_COLS);
                cl.store<C>(cp, ft);
                for (int u = first_u; u < n_units && ok; u += step_u, ++ft.tile) {
                    place(u + step_u);               // (coordinates only)
                    FragTile nxt = ft;
                    if (u + step_u >= n_units) nxt.nc0 = -1;
                    place(u);
                    ok = frag_tile<EPI, ROWS, BNT, PAIR, OUT>(p, cp, ft, nxt, cl, job, release_region);
                }
            }
        } else
        for (int u = first_u; u < n_units && ok; u += step_u) {
            const int64_t m0 = (int64_t)tile_m(u) * BM;
            const int nc0 = tile_n(u) * BN + cgrp * EPI_COLS;    // this warp's first column
            __syncwarp();
#pragma unroll
            for (int h = 0; h < (EPI_COLS + 31) / 32; ++h) {
                const int c = lane + 32 * h;
                if (c >= EPI_COLS) break;
                const int n = nc0 + c < p.N ? nc0 + c : p.N - 1;
                float4 k;
                k.x = __ldg(p.s_w + (int64_t)n * 2) * p.g[0].inv_levels;
                k.y = __ldg(p.s_w + (int64_t)n * 2 + 1) * p.g[1].inv_levels;
                k.z = __int_as_float(p.g[0].center ? p.g[0].center * __ldg(p.colsum + (int64_t)n * 2) : 0);
                k.w = __int_as_float(p.g[1].center ? p.g[1].center * __ldg(p.colsum + (int64_t)n * 2 + 1) : 0);
                colc[c] = k;
            }
            __syncwarp();
            const int64_t m = m0 + row;
            float sa0 = 0.0f, sa1 = 0.0f;
            if (m < p.M) {
                sa0 = p.s_a_per_row ? __ldg(p.s_a + m * 2) : __ldg(p.s_a);
                sa1 = p.s_a_per_row ? __ldg(p.s_a + m * 2 + 1) : __ldg(p.s_a + 1);
            }
            // part: the exact accumulator of the first group (or the running
            // sum of the segments of the tile's only group)
            int32_t part[EPI_COLS];
#pragma unroll
            for (int j = 0; j < EPI_COLS; ++j) part[j] = 0;
            const int gA = g_first, gB = 1 - g_first;
            const int nA = p.g[gA].stages > 0 ? p.g[gA].n_seg : 0;
            const int nB = p.g[gB].stages > 0 ? p.g[gB].n_seg : 0;
            const int njobs = nA + nB;
            const int g_last = nB > 0 ? gB : gA;        // group of the final job
            const bool part_is_other = nA > 0 && nB > 0;
#pragma unroll 1
            for (int jj = 0; jj < njobs; ++jj, ++job) {
                const uint32_t r = job & 1u, use = job >> 1;
                if (!__all_sync(0xffffffffu, wait_bounded(bar(BAR_REG_FULL + r), use & 1u, abort_flag, kTimeoutNs,
                                                          p.err, kErrWait))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t taddr = lane_base + r * REGION;
                if (jj < njobs - 1) {
                    // accumulate: a whole first group, or a segment
                    const int gj = jj < nA ? gA : gB;
                    const float sc = p.g[gj].acc_scale;
#pragma unroll
                    for (int cc = 0; cc < EPI_COLS / 8; ++cc) {
                        uint32_t v[8];
                        tmem_ld8(taddr + cc * 8, v);
#pragma unroll
                        for (int q = 0; q < 8; ++q) part[cc * 8 + q] += __float2int_rn(__uint_as_float(v[q]) * sc);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) release_region(r);
                    if (jj == nA - 1 && part_is_other) {
                        // the first group is complete: add back its centring
#pragma unroll
                        for (int j = 0; j < EPI_COLS; ++j) {
                            const float4 k = colc[j];
                            part[j] += __float_as_int(gA == 0 ? k.z : k.w);
                        }
                    }
                    continue;
                }
                // the final job: finish the tile's outputs, 8 columns at a time
                const float sc = p.g[g_last].acc_scale;
                const bool dbg = p.acc_dbg != nullptr && m < p.M;
                constexpr bool has_next = EPI == EPI_GENERAL_NEXT;
                const bool y_tma = p.y_tma != 0;
                const bool write_y = p.write_y != 0;
                // fp16 outputs go through the staging tile for the TMA store and
                // for the next layer's quantizer
                const bool staged_out = y_tma || has_next;
                if (staged_out) {
                    // the previous tile's store must have read the staging buffer
                    if (lane == 0) bulk_wait_read0();
                    __syncwarp();
                }
#pragma unroll
                for (int cc = 0; cc < EPI_COLS / 8; ++cc) {
                    uint32_t v[8];
                    tmem_ld8(taddr + cc * 8, v);
                    const int nb = nc0 + cc * 8;
                    float y[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int j = cc * 8 + q;
                        const float4 k = colc[j];
                        const int32_t x = __float2int_rn(__uint_as_float(v[q]) * sc) +
                                          __float_as_int(g_last == 0 ? k.z : k.w);
                        const int32_t last = part_is_other ? x : part[j] + x;     // the final job's group
                        const int32_t other = part_is_other ? part[j] : 0;
                        const int32_t a0 = g_last == 0 ? last : other;
                        const int32_t a1 = g_last == 0 ? other : last;
                        y[q] = fmaf(sa1 * k.y, (float)a1, sa0 * k.x * (float)a0);
                        if (dbg && nb + q < p.N) {
                            p.acc_dbg[m * p.N + nb + q] = a0;
                            p.acc_dbg[(p.M + m) * p.N + nb + q] = a1;
                        }
                    }
                    if (staged_out) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if (p.out_bf16) {
                                __nv_bfloat162 h2 = __floats2bfloat162_rn(y[2 * e], y[2 * e + 1]);
                                w[e] = *reinterpret_cast<uint32_t*>(&h2);
                            } else {
                                __half2 h2 = __floats2half2_rn(y[2 * e], y[2 * e + 1]);
                                w[e] = *reinterpret_cast<uint32_t*>(&h2);
                            }
                        }
                        // box cc / 8 (64 columns), row `lane`, 16-byte chunk cc % 8, 128-byte swizzle
                        // (the TMA store map's layout); with 8-column boxes, box cc of 32 x 16 bytes
                        const uint32_t dst =
                            BOX8 ? out_s + (uint32_t)cc * 512u + (uint32_t)lane * 16u
                                 : out_s + (uint32_t)(cc >> 3) * 4096u + (uint32_t)lane * 128u +
                                       ((((uint32_t)cc & 7u) ^ ((uint32_t)lane & 7u)) << 4);
                        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]),
                                     "r"(w[2]), "r"(w[3])
                                     : "memory");
                    }
                    if (write_y && !y_tma && m < p.M) store_out8(p, m, nb, y);
                }
                tc_fence_before();
                if (staged_out) fence_proxy_async_shared();
                __syncwarp();
                if (lane == 0) {
                    release_region(r);
                    if (y_tma && write_y) {
                        // rows and columns beyond M and N are clipped by the store
                        if constexpr (BOX8) {
#pragma unroll
                            for (int bx = 0; bx < EPI_COLS / 8; ++bx)
                                tma_store_2d(&p.tma_y, nc0 + bx * 8, (int)(m0 + quad * 32), out_s + bx * 512u);
                        } else {
#pragma unroll
                            for (int bx = 0; bx < EPI_COLS / 64; ++bx)
                                tma_store_2d(&p.tma_y, nc0 + bx * 64, (int)(m0 + quad * 32), out_s + bx * 4096u);
                        }
                        bulk_commit();
                    }
                }
                if constexpr (has_next) {
                    if (m < p.M) next_layer_codes(p, out_s, lane, m, nc0);
                }
            }
        }
        if (OUT != OUT_BATCH && p.y_tma && p.write_y && lane == 0) bulk_wait0();   // stores complete before the CTA exits
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // the peer's MMAs read this CTA's stages and its commits arrive on this CTA's barriers until it is done
    if constexpr (PAIR) cluster_sync();
    if (warp == WARP_MMA) {
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// 2-D map over expanded rows [rows][row_bytes] with a box of one 128-byte
// K-stage by box_rows rows, 128-byte swizzle (the layout the MMA descriptors read).
bool encode_rows(EncodeTiledFn enc, CUtensorMap* map, const uint8_t* base, int64_t row_bytes, int64_t rows,
                 int box_rows) {
    cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
    cuuint32_t box[2] = {(cuuint32_t)KSTAGE, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, KSTAGE == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- kernel variants ---------------------------------------------------------

struct Variant {
    int epi;
    bool rows;       // LEAN, NEXT: activation scales per row; RUNS: writes debug accumulators (runs_tile's DBG)
    bool f4;
    int bn;
    bool pair;
    int out;
    int smem;
    void (*fn)(SParams);
};

template <int EPI, bool ROWS, int BNT, bool PAIR, int OUT>
constexpr Variant make_variant() {
    return Variant{EPI, ROWS, BNT == BN_F4, BNT, PAIR, OUT, Cfg<BNT, PAIR, OUT>::SMEM_ALLOC,
                   staged_mma_kernel<EPI, ROWS, BNT, PAIR, OUT>};
}

const Variant kVariants[] = {
    make_variant<EPI_LEAN, false, 256, true, OUT_BATCH>(),  make_variant<EPI_LEAN, true, 256, true, OUT_BATCH>(),
    make_variant<EPI_LEAN, false, 256, false, OUT_BATCH>(), make_variant<EPI_LEAN, true, 256, false, OUT_BATCH>(),
    make_variant<EPI_LEAN, false, 256, false, OUT_TMA>(),   make_variant<EPI_LEAN, true, 256, false, OUT_TMA>(),
    make_variant<EPI_LEAN, false, 128, false, OUT_BATCH>(), make_variant<EPI_LEAN, true, 128, false, OUT_BATCH>(),
    make_variant<EPI_LEAN, false, 64, false, OUT_BATCH>(),  make_variant<EPI_LEAN, true, 64, false, OUT_BATCH>(),
    make_variant<EPI_LEAN, false, 240, true, OUT_BATCH>(),  make_variant<EPI_LEAN, true, 240, true, OUT_BATCH>(),
    make_variant<EPI_LEAN, false, 240, false, OUT_BATCH>(), make_variant<EPI_LEAN, true, 240, false, OUT_BATCH>(),
    make_variant<EPI_SEG, true, 256, true, OUT_BATCH>(),    make_variant<EPI_SEG, true, 256, false, OUT_BATCH>(),
    make_variant<EPI_SEG, true, 128, false, OUT_BATCH>(),   make_variant<EPI_SEG, true, 240, true, OUT_BATCH>(),
    make_variant<EPI_SEG, true, 240, false, OUT_BATCH>(),   make_variant<EPI_NEXT, false, 256, false, OUT_TMA>(),
    make_variant<EPI_NEXT, true, 256, false, OUT_TMA>(),    make_variant<EPI_NEXT_SEG, true, 256, false, OUT_TMA>(),
    make_variant<EPI_RUNS, false, 128, false, OUT_BATCH>(), make_variant<EPI_RUNS, false, 64, false, OUT_BATCH>(),
    make_variant<EPI_RUNS, true, 64, false, OUT_BATCH>(),   make_variant<EPI_GENERAL, true, 256, false, OUT_GENERAL>(),
    make_variant<EPI_GENERAL, true, 240, false, OUT_GENERAL>(),
    make_variant<EPI_GENERAL_NEXT, true, 256, false, OUT_GENERAL>(),
};
constexpr int kNumVariants = (int)(sizeof(kVariants) / sizeof(kVariants[0]));

// SM cycles of one tile: max(stages * stage + fixed, epilogue).  Fitted to timed calls
// (one GB300, 1.93 GHz; M x K x N, variant: us): 8192 x 4096 x 4096 pair 109, 256 120,
// 256 TMA 132, 128 156, 64 259; 16384 x 768 x 3072 pair 82, 256 73, 256 TMA 66, 128 79,
// 64 117; 2048 x 4096 x 11008 pair 83, 256 92, 128 116; 512 x 4096 x 4096 pair 28, 256 26,
// 128 23, 64 31; 300 x 4096 x 1024 pair 23, 256 21, 128 17, 64 16.  (An MMA takes about 110
// cycles however narrow, so 64 columns pay only where 128 leave SMs idle.)  There is no term of
// its own for a scale run's drain or for E2M1 stages: those layouts choose by the same costs, unfitted.
struct TileCost {
    double stage, fixed, epilogue;
};
TileCost tile_cost(const Variant& v) {
    if (v.pair) return {560.0, 2500.0, 11500.0};
    if (v.bn > 128) return v.out == OUT_TMA ? TileCost{700.0, 2300.0, 8800.0} : TileCost{640.0, 2500.0, 10200.0};
    if (v.bn > 64) return {420.0, 1800.0, 5000.0};
    return {400.0, 1200.0, 3500.0};
}

// The variant of an epilogue with the shortest modelled time, whole waves of
// tiles; tma: outputs can leave by TMA stores.
const Variant* pick_variant(int epi, bool rows, bool f4, bool tma, int64_t M, int64_t N, int stages) {
    const Variant* best = nullptr;
    double best_t = 0.0;
    for (const Variant& v : kVariants) {
        if (v.epi != epi || v.f4 != f4) continue;
        if ((epi == EPI_LEAN || epi == EPI_NEXT || epi == EPI_RUNS) && v.rows != rows) continue;
        if (epi == EPI_LEAN && v.out == OUT_TMA && !tma) continue;
        const int64_t mt = (M + BM - 1) / BM, nt = (N + v.bn - 1) / v.bn;
        const int64_t slots = v.pair ? num_sms() / 2 : num_sms();
        const int64_t units = v.pair ? (mt + 1) / 2 * nt : mt * nt;
        const int64_t waves = (units + slots - 1) / (slots > 0 ? slots : 1);
        const TileCost c = tile_cost(v);
        const double mma = stages * c.stage + c.fixed;
        const double t = (double)waves * (mma > c.epilogue ? mma : c.epilogue);
        if (best == nullptr || t < best_t) {
            best = &v;
            best_t = t;
        }
    }
    return best;
}

int64_t align1k(int64_t x) { return (x + 1023) / 1024 * 1024; }

}  // namespace staged

bool staged_plan(const LayoutGeom& geo, StagedPlan* sp, bool allow_f4) {
    int nseg_groups = 0;
    int64_t x0 = 0;
    sp->seg_group = -1;
    sp->f4 = 0;
    const bool runs = geo.sub_k > 0;
    // E2M1 pays where its groups hold most of the K codes: the 240-column tiles
    // it needs cost the other group (measured on the 8192 x 4096 x 4096 sweep:
    // +20 % with all codes in E2M1 groups, +6 % at 75 %, -5 % at 50 %)
    if (allow_f4) {
        int64_t f4_codes = 0, all_codes = 0;
        for (int g = 0; g < 2; ++g) {
            const GroupGeom& G = geo.g[g];
            all_codes += G.pw;
            if (G.bits_a <= 2 && G.bits_w <= 2 && geo.act_kind[g] == SONIQ_ACT_UNSIGNED && !runs && G.count > 0)
                f4_codes += G.pw;
        }
        if (f4_codes * 5 < all_codes * 3) allow_f4 = false;
        // and where K is long enough for the MMAs to dominate: at K = 768 (the
        // 16384 x 768 -> 3072 MLP layer) the tile's epilogue sets the pace, and
        // the 240-column epilogue (120 columns per warp, 8-column store boxes)
        // was 10 % slower than the 256-column one
        if (all_codes < 2048) allow_f4 = false;
    }
    for (int g = 0; g < 2; ++g) {
        const GroupGeom& G = geo.g[g];
        StagedGroup& S = sp->g[g];
        const int ak = geo.act_kind[g];
        S.kind = (G.bits_a <= 4 && G.bits_w <= 4) ? 0 : 1;
        // E2M1 holds 0, 0.5, 1, 1.5, 2: codes u <= 3 and |j| <= 2 are exact as code / 2
        if (allow_f4 && G.bits_a <= 2 && G.bits_w <= 2 && ak == SONIQ_ACT_UNSIGNED && !runs && G.count > 0) {
            S.kind = 2;
            sp->f4 = 1;
        }
        // E2M1 rows: two codes per byte, padded to whole 256-code stages
        const int64_t bytes = S.kind == 2 ? (((int64_t)G.pw + 255) / 256 * 256) / 2
                                          : (int64_t)G.pw * (S.kind == 0 ? 1 : 2);
        S.stages = (int32_t)(bytes / staged::KSTAGE);
        S.x0 = (int32_t)x0;
        x0 += bytes;
        // unsigned fp16 activations are centred (halving the products) unless every
        // run is scaled on its own, where the centring's weight sums would be per run
        S.center = (S.kind == 1 && ak == SONIQ_ACT_UNSIGNED && !runs) ? (1 << (G.bits_a - 1)) : 0;
        const int64_t amax = ak == SONIQ_ACT_PM1 ? 1
                                                 : (ak == SONIQ_ACT_SIGNED || S.center ? (int64_t)1 << (G.bits_a - 1)
                                                                                       : (1 << G.bits_a) - 1);
        const int64_t wmax = ak == SONIQ_ACT_PM1 ? 1 : (int64_t)1 << (G.bits_w - 1);
        const int64_t maxprod = amax * wmax;
        const int64_t codes_per_stage = S.kind == 2 ? 2 * staged::KSTAGE : (S.kind == 0 ? staged::KSTAGE : staged::KSTAGE / 2);
        int64_t seg_stages = ((int64_t)1 << 24) / maxprod / codes_per_stage;
        if (runs) {
            // one job per run; its exact sum must stay within 2^24
            if ((int64_t)geo.sub_k * maxprod > ((int64_t)1 << 24)) return false;
            seg_stages = geo.sub_k / codes_per_stage;
        }
        if (seg_stages < 1) return false;
        S.seg_stages = (int32_t)(seg_stages < S.stages ? seg_stages : (S.stages > 0 ? S.stages : 1));
        S.n_seg = S.stages > 0 ? (S.stages + S.seg_stages - 1) / S.seg_stages : 0;
        if (S.n_seg > 1 && !runs) {
            ++nseg_groups;
            sp->seg_group = g;
        }
    }
    if (nseg_groups > 1) return false;
    sp->eb = x0;
    return x0 > 0 && x0 % 128 == 0;
}

int64_t staged_scratch_bytes(const LayoutGeom& geo, int64_t rows_a, int64_t N) {
    StagedPlan sp;
    if (!staged_plan(geo, &sp)) return 0;
    return staged::align1k(rows_a * sp.eb) + staged::align1k(N * sp.eb) + staged::align1k(N * 8);
}

cudaError_t launch_staged(const LayoutGeom& geo, const MmaArgs& a, void* scratch, size_t scratch_bytes,
                          cudaStream_t st) {
    using namespace staged;
    StagedPlan sp;
    // E2M1 groups need 240-column tiles: not with a next layer (its codes are
    // packed from 64-column output boxes), nor where the narrower tiles would
    // add more than 7 % of padded columns (N = 256 would take two tiles)
    const bool f4_ok = a.next == nullptr && (int64_t)((a.N + BN_F4 - 1) / BN_F4) * BN_F4 * 100 <= (int64_t)a.N * 107;
    if (!staged_plan(geo, &sp, f4_ok)) return cudaErrorNotSupported;
    const int64_t rows_a = a.M;
    if ((int64_t)scratch_bytes < staged_scratch_bytes(geo, rows_a, a.N) || scratch == nullptr ||
        (uintptr_t)scratch % 256 != 0)
        return cudaErrorNotSupported;
    uint8_t* xa = static_cast<uint8_t*>(scratch);
    uint8_t* xw = xa + align1k(rows_a * sp.eb);
    int32_t* colsum = reinterpret_cast<int32_t*>(xw + align1k((int64_t)a.N * sp.eb));

    // ---- expand activations (im2col for a convolution) and weights ----
    ExpandParams e;
    memset(&e, 0, sizeof(e));
    for (int g = 0; g < 2; ++g) {
        const GroupGeom& G = geo.g[g];
        e.bits[g] = G.bits_a;
        e.kind[g] = sp.g[g].kind;
        e.src_off[g] = G.a_off;
        e.dst_off[g] = sp.g[g].x0;
        e.blk_src[g] = G.pa / 32;
        // E2M1 groups are written out to whole 256-code stages (zero codes)
        e.blk_dst[g] = (sp.g[g].kind == 2 ? (G.pw + 255) / 256 * 256 : G.pw) / 32;
        e.center[g] = sp.g[g].center;
        e.cpt[g] = G.pa / 32 > 0 ? G.pa / 32 : 1;
        e.cpt_magic[g] = (((uint64_t)1 << 32) + (uint64_t)e.cpt[g] - 1) / (uint64_t)e.cpt[g];
        // a block's parts start at multiples of 8 bytes where its words come in pairs (4-bit slices)
        e.vec8[g] = (G.a_off % 8 == 0 && geo.a_row_bytes % 8 == 0 && (uintptr_t)a.Ap % 8 == 0 && G.bits_a % 2 == 0) ? 1 : 0;
        e.code_kind[g] = geo.act_kind[g];
        e.count[g] = G.count;
    }
    e.src = a.Ap;
    e.src_row_bytes = geo.a_row_bytes;
    e.dst = xa;
    e.dst_row_bytes = sp.eb;
    e.rows = rows_a;
    e.is_weight = 0;
    e.conv = a.conv;
    e.H = a.H; e.W = a.W; e.P = a.P; e.Q = a.Q; e.R = a.R; e.S = a.S;
    e.sh = a.sh; e.sw = a.sw; e.ph = a.ph; e.pw = a.pw;
    auto grid_for = [](int64_t items) {
        int64_t ctas = (items + 7) / 8;                        // 8 warps per CTA, one (four rows, group) per warp
        const int64_t cap = (int64_t)num_sms() * 16;
        return (int)(ctas < 1 ? 1 : (ctas > cap ? cap : ctas));
    };
    ExpandParams w = e;
    for (int g = 0; g < 2; ++g) {
        const GroupGeom& G = geo.g[g];
        w.bits[g] = G.bits_w;
        w.src_off[g] = G.w_off;
        w.blk_src[g] = G.pw / 32;
        w.center[g] = 0;
        w.vec8[g] = (G.w_off % 8 == 0 && geo.w_row_bytes % 8 == 0 && (uintptr_t)a.Wp % 8 == 0 && G.bits_w % 2 == 0) ? 1 : 0;
        w.code_kind[g] = geo.act_kind[g] == SONIQ_ACT_PM1 ? 2 : 1;
    }
    w.src = a.Wp;
    w.src_row_bytes = geo.w_row_bytes;
    w.dst = xw;
    w.rows = a.N;
    w.is_weight = 1;
    w.colsum = colsum;
    w.conv = 0;
    // activations and weights in one launch
    cudaError_t err = cudaSuccess;
    if (!launch_stream(e, w, st, &err))
        err = launch_pdl(expand_kernel,
                         dim3((unsigned)grid_for((rows_a + kExpandRows - 1) / kExpandRows * 2 +
                                                 ((int64_t)a.N + kExpandRows - 1) / kExpandRows * 2)),
                         dim3(256), 0, st, e, w);
    note_launch();
    if (err != cudaSuccess) return err;

    // ---- the GEMM ----
    SParams p;
    memset(&p, 0, sizeof(p));
    EncodeTiledFn enc = encode_fn();
    if (enc == nullptr) return cudaErrorNotSupported;
    // ---- epilogue, tile width and pairing ----
    const bool runs = geo.sub_k > 0, wr_y = a.Y != nullptr, has_next = a.next != nullptr;
    const bool general = !runs && (a.acc_dbg != nullptr || (!wr_y && !has_next) ||
                                   (a.flags & SONIQ_FLAG_TEST_DROP_ARRIVE) != 0);
    const int epi = runs ? EPI_RUNS
                    : general ? (has_next ? EPI_GENERAL_NEXT : EPI_GENERAL)
                    : has_next ? (sp.seg_group >= 0 ? EPI_NEXT_SEG : EPI_NEXT)
                    : sp.seg_group >= 0 ? EPI_SEG : EPI_LEAN;
    const Variant* var = pick_variant(epi, runs ? a.acc_dbg != nullptr : a.s_a_per_row != 0, sp.f4 != 0, wr_y && a.N % 8 == 0,
                                      a.M, a.N, (int)(sp.eb / KSTAGE));
    if (var == nullptr) return cudaErrorNotSupported;
    const int tile_n = var->bn;
    const bool pair = var->pair;
    if (!encode_rows(enc, &p.tma_a, xa, sp.eb, rows_a, BM) ||
        !encode_rows(enc, &p.tma_b, xw, sp.eb, a.N, pair ? tile_n / 2 : tile_n))
        return cudaErrorInvalidValue;
    p.s_a = a.s_a;
    p.s_w = a.s_w;
    p.colsum = colsum;
    p.Y = a.Y;
    p.acc_dbg = a.acc_dbg;
    p.err = device_error_word();
    if (p.err == nullptr) return cudaErrorUnknown;
    p.M = a.M;
    p.N = a.N;
    p.m_tiles = (int32_t)((a.M + BM - 1) / BM);
    p.n_tiles = (a.N + tile_n - 1) / tile_n;
    p.total_tiles = p.m_tiles * p.n_tiles;
    p.s_a_per_row = a.s_a_per_row;
    p.out_bf16 = a.out_bf16;
    p.seg_group = sp.seg_group;
    p.drop_first = (a.flags & SONIQ_FLAG_TEST_DROP_ARRIVE) != 0 ? 1 : 0;
    p.write_y = a.Y != nullptr;
    if (a.next != nullptr) {
        p.has_next = 1;
        p.s_next = a.next_s_a;
        p.Ap_next = a.next_Ap;
        p.next_row_bytes = a.next->a_row_bytes;
        p.next_pa0 = a.next->g[0].pa;
        for (int g = 0; g < 2; ++g) {
            p.next_count[g] = a.next->g[g].count;
            p.next_bits[g] = a.next->g[g].bits_a;
            p.next_off[g] = a.next->g[g].a_off;
        }
    }
    // outputs through TMA stores when the row pitch allows a tensor map (N * 2 bytes a multiple of 16)
    p.y_tma = 0;
    if (var->out != OUT_BATCH && p.write_y && a.N % 8 == 0 && (uintptr_t)a.Y % 16 == 0) {
        cuuint64_t dims[2] = {(cuuint64_t)a.N, (cuuint64_t)a.M};
        cuuint64_t strides[1] = {(cuuint64_t)a.N * 2};
        // 64 x 32 boxes, 128-byte swizzled, where a warp's columns are whole boxes; else 8 x 32 boxes
        const bool box8 = tile_n / (NUM_EPI_WARPS / 4) % 64 != 0;
        cuuint32_t box[2] = {box8 ? 8u : 64u, 32u};
        cuuint32_t estr[2] = {1, 1};
        if (enc(&p.tma_y, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, a.Y, dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, box8 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        p.y_tma = 1;
    }
    for (int g = 0; g < 2; ++g) {
        const GroupGeom& G = geo.g[g];
        SGroup& S = p.g[g];
        S.kind = sp.g[g].kind;
        S.stages = sp.g[g].stages;
        S.x0 = sp.g[g].x0;
        S.seg_stages = sp.g[g].seg_stages;
        S.n_seg = sp.g[g].n_seg;
        S.center = sp.g[g].center;
        S.acc_scale = S.kind == 0 ? 262144.0f : (S.kind == 2 ? 4.0f : 1.0f);   // 2^18, 1, or 4 (products u j / 4)
        // decode levels: activations 2^na - 1 (unsigned), 2^(na-1) (signed) or 1 (+-1);
        // weights 2^(nw-1) or 1 (+-1)
        const int ak = geo.act_kind[g];
        const double la = ak == SONIQ_ACT_PM1 ? 1.0 : (ak == SONIQ_ACT_SIGNED ? (double)(1 << (G.bits_a - 1))
                                                                             : (double)((1 << G.bits_a) - 1));
        const double lw = ak == SONIQ_ACT_PM1 ? 1.0 : (double)(1 << (G.bits_w - 1));
        S.inv_levels = (float)(1.0 / (la * lw));
    }
    p.runs = runs ? 1 : 0;
    p.nb = geo.nb;
    p.pair_tiles = ((p.m_tiles + 1) / 2) * p.n_tiles;
    static bool attr_done[64][kNumVariants] = {};
    static int max_pairs[64][kNumVariants] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    const int kidx = (int)(var - kVariants);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.blockDim = dim3(NUM_THREADS, 1, 1);
    cfg.dynamicSmemBytes = var->smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (!attr_done[dev][kidx]) {
        if ((err = cudaFuncSetAttribute((const void*)var->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, var->smem)) !=
            cudaSuccess)
            return err;
        if ((err = prefer_max_shared((const void*)var->fn)) != cudaSuccess) return err;
        if (pair) {
            // pairs that can be resident at once (one CTA per SM)
            cfg.gridDim = dim3(2 * (unsigned)num_sms() / 2, 1, 1);
            int n = 0;
            if ((err = cudaOccupancyMaxActiveClusters(&n, (const void*)var->fn, &cfg)) != cudaSuccess) return err;
            max_pairs[dev][kidx] = n;
        }
        attr_done[dev][kidx] = true;
    }
    if (pair) {
        int pairs = max_pairs[dev][kidx];
        if (pairs < 1) return cudaErrorNotSupported;
        if (pairs > p.pair_tiles) pairs = p.pair_tiles;
        cfg.gridDim = dim3(2 * (unsigned)pairs, 1, 1);
        cfg.numAttrs = 2;
        if ((err = cudaLaunchKernelEx(&cfg, var->fn, p)) != cudaSuccess) return err;
    } else {
        const int grid = p.total_tiles < num_sms() ? p.total_tiles : num_sms();
        if ((err = launch_pdl(var->fn, dim3((unsigned)grid), dim3(NUM_THREADS), (size_t)var->smem, st, p)) !=
            cudaSuccess)
            return err;
    }
    note_launch();
    return cudaGetLastError();
}

}  // namespace soniq

// Tiled activation quantize-and-pack with bulk-staged rows: Sec. 3
// "Enabling Low-Cost Fixed-Point Operations" step 2 (unsigned codes) with the
// channel permutation and padding of Sec. 4.1.
//
// A persistent CTA (one per SM) streams tiles of TR consecutive rows.  A
// producer warp copies each row of a tile into a ring of shared-memory stages
// with one bulk copy (rows stay in their original channel order; a 16-byte
// zero slot after every row stands in for the padding positions); a stage is
// refilled as soon as the consumer warps (up to 20, as many as the layout's
// block ranges need) have released it through its "empty" mbarrier, so no
// CTA-wide barrier sits in the tile loop.  Codes are formed one lane per
// packed position: each consumer warp owns a contiguous range of whole
// 8-block chunks of one precision group (its quantizer constants are
// warp-uniform) and, where warps are left over, a share of the tile's rows;
// it holds the staged-row byte offsets of its lanes' channels and walks its
// rows with up to 8 independent gathers per row, so every gather instruction
// reads one row (conflict-free where the permutation keeps channels in order,
// as it does within each group).  The code lands as
// one byte in a per-tile code buffer; after a warp barrier each lane packs
// whole 32-code blocks of that warp and stores them with 16-byte stores.
//
// The code of Sec. 3 step 2, u = clip(rint(RN(RN(a / s) * (2^n - 1))), 0,
// 2^n - 1): the quotient by Markstein's correction step (scales in
// [2^-60, 2^60], exact as in the other quantize kernels), IEEE division
// otherwise; the clip is taken before rounding (its bounds are integers, so
// clip and rint commute), on the quotient (saturated to [0, 1], NaN to 0); rint is
// the addition of 1.5 * 2^23, after which the low byte of the sum's bits is
// the integer.  Under a calibrated scale the top clip is taken on the input
// instead (a above s becomes s, whose quotient is exactly 1): +inf then
// gets the top code, where the residual step would have made it NaN.
//
// Scale modes: given scales (per tensor after the separate absmax pass, or
// calibrated), per (row, group) maxima found from the staged rows, or per-tensor
// maxima found in a first pass over the rows, with a grid barrier.
#include <cuda_fp16.h>

#include <type_traits>

#include "soniq_device.cuh"
#include "soniq_internal.h"
#include "tc_ptx.cuh"

namespace soniq {
namespace {

constexpr int kGatherConsumerWarps = 20;                    // at most, code-forming warps
constexpr int kGatherMinConsumerWarps = 8;                  // per-row maxima: one warp per tile row
constexpr int kGatherThreads = (kGatherConsumerWarps + 1) * 32;   // + one producer warp
constexpr int kGatherMaxRows = 8;        // rows of a tile per warp
constexpr int kGatherMaxStages = 6;      // tiles in the ring (all but one in flight)
constexpr size_t kGatherSmemBudget = 220 * 1024;

struct GatherParams {
    const uint16_t* A;
    uint8_t* Ap;
    float* s_a;              // [2] in (given scales) or [M][2] out (per row)
    const int32_t* perm;
    unsigned* err;
    long long timeout_ns;
    int64_t M;
    int32_t K;
    int32_t a_row_bytes;
    int32_t demote;          // reset the L2 eviction priority of every input line read
    int32_t tile_rows;
    int32_t stages;
    int32_t row_stride;      // bytes between staged rows (2K + 16, rounded up to 16)
    int32_t nblk0, nblk;     // 32-code blocks of group 0 / of both groups per row
    int32_t bpw;             // 32-code blocks per warp; each warp takes blocks of one group
    int32_t w0;              // block ranges 0 .. w0-1 are of group 0, w0 .. wb-1 of group 1
    int32_t wb;              // block ranges
    int32_t rg;              // row groups: warp w takes range w % wb and rows w / wb, + rg, ...
    int32_t nwc;             // consumer warps (the producer is warp nwc)
    // MODE 3: grid barrier (arrivals, generation) and per-CTA maxima [grid][2]
    unsigned* bar;
    float* part;
    unsigned err_bit;
    int32_t drop_arrival;
    GroupGeom g[2];
};

// Shared-memory accesses with explicit 32-bit shared addresses.  The load is
// not volatile, so the compiler may schedule the gathers of a row together;
// its address derives from a base that fresh() hands out after the stage's
// wait, which keeps it behind that wait.
__device__ __forceinline__ float lds_half(uint32_t addr) {
    uint16_t v;
    asm("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return __half2float(__ushort_as_half(v));
}

__device__ __forceinline__ void sts_u8(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t fresh(uint32_t v) {
    uint32_t r;
    asm volatile("mov.b32 %0, %1;" : "=r"(r) : "r"(v) : "memory");
    return r;
}

// Bits of 1.5 * 2^23 + rint(clip(RN(q * levels), 0, levels)); the low byte is the code.
__device__ __forceinline__ uint32_t code_bits(float q, float levels) {
    float t = __fmul_rn(q, levels);
    t = fminf(fmaxf(t, 0.0f), levels);
    return __float_as_uint(__fadd_rn(t, 12582912.0f));
}

// Quantizer of one (tensor or row, group): mode 1 Markstein quotient, 2 IEEE
// division, 0 every code 0 (no positive scale).
struct GConst {
    float s, r, levels;
    int mode;
};

__device__ __forceinline__ GConst gconst(float s, int bits) {
    GConst k;
    k.s = s;
    k.levels = (float)((1 << bits) - 1);
    k.mode = (s >= 0x1p-60f && s <= 0x1p60f) ? 1 : (s > 0.0f ? 2 : 0);
    k.r = k.mode == 1 ? __frcp_rn(s) : 0.0f;
    return k;
}

__device__ __forceinline__ uint32_t quant_one(float a, const GConst& k) {
    float q;
    if (k.mode == 1) {
        const float q0 = __fmul_rn(a, k.r);
        q = __fmaf_rn(__fmaf_rn(-q0, k.s, a), k.r, q0);
    } else {
        q = k.mode == 2 ? __fdiv_rn(a, k.s) : 0.0f;
    }
    return code_bits(q, k.levels);
}

// Per-group max |a| of one staged row (original channel order; grp_s holds
// 0xFFFF in the halves of group-1 channels), by one warp.
__device__ __forceinline__ void row_group_max(const uint8_t* row, const uint32_t* grp_s, int K, float& f0, float& f1) {
    const int lane = threadIdx.x & 31;
    __half2 g0 = __float2half2_rn(0.0f), g1 = g0;
    for (int v = lane; v < K / 8; v += 32) {
        const uint4 x = reinterpret_cast<const uint4*>(row)[v];
        const uint4 m = *reinterpret_cast<const uint4*>(grp_s + 4 * v);
        const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, mw[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // |a| (sign cleared) of the group's halves, 0 elsewhere; fp16 max drops NaN
            uint32_t a1 = xw[q] & mw[q] & 0x7FFF7FFFu, a0 = xw[q] & ~mw[q] & 0x7FFF7FFFu;
            g1 = __hmax2(g1, *reinterpret_cast<__half2*>(&a1));
            g0 = __hmax2(g0, *reinterpret_cast<__half2*>(&a0));
        }
    }
    f0 = fmaxf(__low2float(g0), __high2float(g0));
    f1 = fmaxf(__low2float(g1), __high2float(g1));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        f0 = fmaxf(f0, __shfl_xor_sync(0xffffffffu, f0, o));
        f1 = fmaxf(f1, __shfl_xor_sync(0xffffffffu, f1, o));
    }
}

}  // namespace

namespace {

// Per packed position: the channel's byte offset in a staged row, or in MODE 3,
// whose kept tiles want the room, the channel in 16 bits.
template <int MODE>
using GatherOff = std::conditional_t<MODE == 3, uint16_t, uint32_t>;

// Codes of nc <= 8 consecutive 32-code blocks of one group (positions pos0 +
// 32 j of this lane) for rows rr0, rr0 + rgs, ... < nr of the tile, into the
// code buffer.  Absent blocks of a short chunk read the zero slot and skip
// their stores.  kc: per-row quantizers (MODE 2), kg: the group's quantizer
// otherwise.
//
// Bound by instruction issue.  Two codes share each packed fp32 instruction,
// and the clip at 0 (and of a NaN) is the saturation of the quotient's last
// step: 6 instructions a code instead of 10.  The rows are a loop of one: with
// all eight unrolled the kernel's instructions came cold for every tile (a
// third of the stalls), with two 2048 x 16384 took 47 us instead of 42.
template <int MODE>
__device__ __forceinline__ void codes_chunk8(uint32_t rows_ba, uint32_t codes_a, const GatherOff<MODE>* offs_s, int pos0, int nc,
                                             int rr0, int rgs, int nr, uint32_t S, int npos, const GConst (*kc)[2],
                                             const GConst& kg, int g, float lv, uint32_t zero_slot) {
    uint32_t off[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) off[j] = j < nc ? (MODE == 3 ? 2u : 1u) * offs_s[pos0 + 32 * j] : zero_slot;
    uint32_t row = rows_ba + (uint32_t)rr0 * S, crow = codes_a + (uint32_t)(rr0 * npos + pos0);
    const float2 lv2 = make_float2(lv, lv);
#pragma unroll 1
    for (int r = rr0; r < nr; r += rgs, row += (uint32_t)rgs * S, crow += (uint32_t)(rgs * npos)) {
        const GConst kk = MODE == 2 ? kc[r][g] : kg;
        if (kk.mode == 1) {
            float a[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) a[j] = lds_half(row + off[j]);
            const float2 r2 = make_float2(kk.r, kk.r), ms2 = make_float2(-kk.s, -kk.s);
            float2 u[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 x = make_float2(a[2 * j], a[2 * j + 1]);
                if (MODE == 0) x = make_float2(fmin_keep_nan(x.x, kk.s), fmin_keep_nan(x.y, kk.s));
                const float2 q0 = mul2(x, r2);
                const float2 e = fma2(q0, ms2, x);
                const float2 q = make_float2(fma_sat(e.x, kk.r, q0.x), fma_sat(e.y, kk.r, q0.y));
                u[j] = add2(mul2(q, lv2), 12582912.0f);
            }
            if (nc == 8) {
#pragma unroll
                for (int j = 0; j < 8; ++j) sts_u8(crow + 32u * j, __float_as_uint((j & 1) ? u[j >> 1].y : u[j >> 1].x));
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j < nc) sts_u8(crow + 32u * j, __float_as_uint((j & 1) ? u[j >> 1].y : u[j >> 1].x));
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j < nc) sts_u8(crow + 32u * j, quant_one(lds_half(row + off[j]), kk));
        }
    }
}

// MODE 0: calibrated scales s_a[2] (codes clip at the top); 1: per-tensor
// scales s_a[2], the group maxima of these same values; 2: per-(row, group)
// maxima found here; 3: per-tensor scales found here (s_a out).  With the
// group maximum as the scale, |a| <= s, so the correctly rounded quotient is
// at most 1 and RN(q * levels) at most levels: the top clip is void in modes
// 1 to 3 (on the Markstein path; the IEEE path, taken for scales outside
// [2^-60, 2^60], keeps it).
//
// MODE 3 runs over the CTA's tiles twice, with a grid barrier in between (a
// cooperative launch).  The first pass folds the group maxima and leaves the
// last tiles in the ring; the second starts with those and then streams the
// earlier ones again, latest first, out of L2.
template <int MODE>
__global__ void __launch_bounds__(kGatherThreads, 1) quantize_gather_kernel(const GatherParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full_bar[kGatherMaxStages], empty_bar[kGatherMaxStages];
    __shared__ uint32_t abort_s, none_s, lost_s, max_s[2];
    __shared__ GConst kc_s[2][kGatherMaxRows][2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int TR = p.tile_rows, NST = p.stages, K = p.K;
    const uint32_t S = (uint32_t)p.row_stride, row_bytes = 2u * (uint32_t)K;
    const int pa0 = p.g[0].pa, npos = pa0 + p.g[1].pa;
    const int c0 = p.g[0].count, c1 = p.g[1].count;
    // shared memory: channels | group masks (MODE 2: per channel; MODE 3: a bit each) | codes | staged rows
    GatherOff<MODE>* offs_s = reinterpret_cast<GatherOff<MODE>*>(smem);
    size_t o = ((size_t)npos * sizeof(GatherOff<MODE>) + 15) & ~(size_t)15;
    uint32_t* grp_s = reinterpret_cast<uint32_t*>(smem + o);
    if (MODE == 2) o += ((size_t)K * 2 + 15) & ~(size_t)15;
    if (MODE == 3) o += ((size_t)K / 8 + 19) & ~(size_t)15;
    uint8_t* codes_s = smem + o;
    o += ((size_t)TR * npos + 15) & ~(size_t)15;
    uint8_t* rows_s = smem + o;
    const uint32_t rows_a = tc::smem_u32(rows_s);
    const uint32_t abort_flag = tc::smem_u32(&abort_s);
    const int64_t ntiles = (p.M + TR - 1) / TR;
    // this CTA's tiles: blockIdx.x + i gridDim.x for i < n; MODE 3 runs over them as
    // ring uses 0 .. n - 1, then the kept ones again in place, then n .. for the others
    const int n = ntiles > blockIdx.x ? (int)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
    const int kept = MODE == 3 ? (n < NST ? n : NST) : 0;
    const int uses = MODE == 3 ? n + (n - kept) : n;
    auto tile_of = [&](int use) {
        const int i = use < n ? use : (n - kept - 1) - (use - n);
        return (int64_t)blockIdx.x + (int64_t)i * gridDim.x;
    };

    if (tid == 0) {
        for (int b = 0; b < NST; ++b) {
            tc::mbar_init(tc::smem_u32(&full_bar[b]), 1);
            tc::mbar_init(tc::smem_u32(&empty_bar[b]), (uint32_t)p.nwc);
        }
        tc::set_flag(abort_flag, 0);
        lost_s = 0u;
        max_s[0] = max_s[1] = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // launched after the previous kernel's start (launch_pdl): every global
    // access comes after this wait; one wave of CTAs, so the kernel that
    // follows may be scheduled at once
    tc::pdl_wait();
    if (MODE != 3) tc::pdl_trigger();

    if (warp == p.nwc) {
        // ---- producer: one lane streams tiles into the stage ring ----
        if (lane == 0) {
            int b = 0;
            uint32_t round = 0u;
            for (int u = 0; u < uses; ++u) {
                // (MODE 3: twice the limit, so that a lost grid barrier is the consumers' to report)
                if (round > 0u &&
                    !tc::wait_bounded(tc::smem_u32(&empty_bar[b]), (round - 1u) & 1u, abort_flag,
                                      MODE == 3 ? 2 * p.timeout_ns : p.timeout_ns, p.err, kErrWait))
                    break;
                const int64_t m0 = tile_of(u) * TR;
                const int nr = p.M - m0 < TR ? (int)(p.M - m0) : TR;
                const uint32_t bar = tc::smem_u32(&full_bar[b]);
                tc::mbar_arrive_expect_tx(bar, (uint32_t)nr * row_bytes);
                for (int r = 0; r < nr; ++r)
                    tc::bulk_load(rows_a + (uint32_t)(b * TR + r) * S, p.A + (m0 + r) * K, row_bytes, bar);
                if (++b == NST) {
                    b = 0;
                    ++round;
                }
            }
            // the copies in flight land before the CTA exits, also when it was abandoned (the abort
            // flag may be up, so these waits get a flag of their own)
            none_s = 0u;
            for (int i = 0; i < NST; ++i) {
                const uint32_t taken = round + (i < b ? 1u : 0u);       // tiles the stage has taken
                if (taken > 0u)
                    tc::wait_bounded(tc::smem_u32(&full_bar[i]), (taken - 1u) & 1u, tc::smem_u32(&none_s), p.timeout_ns,
                                     p.err, kErrWait);
            }
        }
        return;
    }

    // ---- consumers (p.nwc warps) ----
    const int nthr_c = 32 * p.nwc;
    auto consumer_sync = [nthr_c] { asm volatile("bar.sync 1, %0;" ::"r"(nthr_c) : "memory"); };
    if (MODE == 2 || MODE == 3) {
        const int words = MODE == 2 ? K / 2 : (K + 31) / 32;
        for (int w = tid; w < words; w += nthr_c) grp_s[w] = 0u;
        consumer_sync();
    }
    // channels: the permutation's loads issued eight at a time.  The offsets are stored in a
    // loop of their own, the masks marked in another: with both in one loop given scales took
    // 11.1 us for 1 x 16384 (6.9 so), 7.8 for 400 x 8192 (5.5), 21.3 for 8192 x 4096 (19.0).
    for (int q0 = tid; q0 < npos; q0 += 8 * nthr_c) {
        int ch[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = q0 + u * nthr_c;
            int j = -1;
            if (q < pa0) j = q < c0 ? q : -1;
            else if (q < npos) j = q - pa0 < c1 ? c0 + (q - pa0) : -1;
            ch[u] = j >= 0 ? __ldg(p.perm + j) : -1;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = q0 + u * nthr_c;
            // padding: the zero slot
            if (q < npos)
                offs_s[q] = (GatherOff<MODE>)(MODE == 3 ? (ch[u] >= 0 ? ch[u] : K)
                                                        : (ch[u] >= 0 ? 2u * (uint32_t)ch[u] : row_bytes));
        }
        if constexpr (MODE >= 2) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (q0 + u * nthr_c < pa0 || ch[u] < 0) continue;
                if (MODE == 2) atomicOr(grp_s + (ch[u] >> 1), (ch[u] & 1) ? 0xFFFF0000u : 0x0000FFFFu);
                else atomicOr(grp_s + (ch[u] >> 5), 1u << (ch[u] & 31));
            }
        }
    }
    // the zero slot after every staged row (the bulk copies write only the row itself)
    for (int r = tid; r < NST * TR; r += nthr_c)
        *reinterpret_cast<uint4*>(rows_s + (size_t)r * S + row_bytes) = make_uint4(0u, 0u, 0u, 0u);
    consumer_sync();

    // this warp's group, its blocks bw0 .. bw0 + nbw - 1 within the group, and
    // its rows rr0, rr0 + rg, ... of each tile (warps past wb * rg stay idle)
    const bool active = warp < p.wb * p.rg;
    const int wbi = warp % p.wb, rr0 = warp / p.wb, rgs = p.rg;
    const int g = wbi < p.w0 ? 0 : 1;
    const int bw0 = (g ? wbi - p.w0 : wbi) * p.bpw;
    const int nblk_g = g ? p.nblk - p.nblk0 : p.nblk0;
    const int nbw = active ? max(0, min(p.bpw, nblk_g - bw0)) : 0;
    const int gbase = g ? pa0 : 0;
    const int bits = p.g[g].bits_a;
    const int a_off = p.g[g].a_off;
    GConst kg;
    if (MODE == 0 || MODE == 1) kg = gconst(p.s_a[g], bits);
    const float lv = (float)((1 << bits) - 1);

    if (MODE == 3) {
        // ---- group maxima of this CTA's rows: thread -> 16-byte column, rows tr, tr + rp, ... ----
        const int KV = K / 8, cols = KV < nthr_c ? KV : nthr_c, rp = nthr_c / cols;
        const int col = tid % cols, tr = tid / cols;
        __half2 g0 = __float2half2_rn(0.0f), g1 = g0;
        int b = 0;
        uint32_t parity = 0u;
        for (int u = 0; u < n; ++u) {
            const int64_t m0 = tile_of(u) * TR;
            const int nr = p.M - m0 < TR ? (int)(p.M - m0) : TR;
            const bool ok = tc::wait_bounded_warp(tc::smem_u32(&full_bar[b]), parity, abort_flag, p.timeout_ns, p.err,
                                                  kErrWait);
            const uint32_t rows_ba = fresh(rows_a + (uint32_t)(b * TR) * S);
            if (ok && tr < rp) {
                for (int v = col; v < KV; v += cols) {
                    const uint32_t bt = grp_s[v >> 2] >> (8 * (v & 3));    // the vector's eight channels
                    uint32_t m1[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        m1[q] = (bt >> (2 * q) & 1u) * 0x7FFFu | (bt >> (2 * q + 1) & 1u) * 0x7FFF0000u;
                    for (int r = tr; r < nr; r += rp) {
                        uint4 x;
                        asm("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                            : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                            : "r"(rows_ba + (uint32_t)r * S + 16u * (uint32_t)v));
                        const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            // |a| of each group's halves, 0 elsewhere; the fp16 maximum drops NaN
                            uint32_t a1 = xw[q] & m1[q], a0 = xw[q] & (m1[q] ^ 0x7FFF7FFFu);
                            g1 = __hmax2(g1, *reinterpret_cast<__half2*>(&a1));
                            g0 = __hmax2(g0, *reinterpret_cast<__half2*>(&a0));
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0 && u < n - kept) tc::mbar_arrive(tc::smem_u32(&empty_bar[b]));
            if (++b == NST) {
                b = 0;
                parity ^= 1u;
            }
        }
        // non-negative floats order as their bits
        const uint32_t b0 = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(__low2float(g0), __high2float(g0))));
        const uint32_t b1 = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(__low2float(g1), __high2float(g1))));
        if (lane == 0) {
            atomicMax(&max_s[0], b0);
            atomicMax(&max_s[1], b1);
        }
        consumer_sync();
        // ---- grid barrier: the last CTA to arrive resets the count and advances the generation ----
        if (tid == 0) {
            p.part[2 * blockIdx.x] = __uint_as_float(max_s[0]);
            p.part[2 * blockIdx.x + 1] = __uint_as_float(max_s[1]);
            const unsigned gen = *reinterpret_cast<volatile unsigned*>(p.bar + 1);
            __threadfence();
            if (!(p.drop_arrival && blockIdx.x == 0) && !tc::abort_raised(abort_flag) &&
                atomicAdd(p.bar, 1u) == gridDim.x - 1) {
                *reinterpret_cast<volatile unsigned*>(p.bar) = 0u;
                __threadfence();
                atomicAdd(p.bar + 1, 1u);
            }
            long long t0 = 0;
            for (uint32_t it = 0;; ++it) {
                if (*reinterpret_cast<volatile unsigned*>(p.bar + 1) != gen) break;
                if ((it & 63u) == 63u) {
                    const long long t = tc::globaltimer();
                    if (t0 == 0) t0 = t;
                    else if (t - t0 > p.timeout_ns) {
                        atomicOr(p.err, p.err_bit);
                        lost_s = 1u;
                        tc::set_flag(abort_flag, 1);       // the producer stops waiting
                        break;
                    }
                }
            }
            __threadfence();
        }
        consumer_sync();
        if (lost_s) return;
        tc::pdl_trigger();
        // every warp folds all CTAs' maxima
        uint32_t s0 = 0u, s1 = 0u;
        for (int i = lane; i < (int)gridDim.x; i += 32) {
            const float2 v = __ldcg(reinterpret_cast<const float2*>(p.part) + i);
            s0 = max(s0, __float_as_uint(v.x));
            s1 = max(s1, __float_as_uint(v.y));
        }
        s0 = __reduce_max_sync(0xffffffffu, s0);
        s1 = __reduce_max_sync(0xffffffffu, s1);
        if (blockIdx.x == 0 && tid == 0) {
            p.s_a[0] = __uint_as_float(s0);
            p.s_a[1] = __uint_as_float(s1);
        }
        kg = gconst(__uint_as_float(g ? s1 : s0), bits);
    }

    const uint8_t* A8 = reinterpret_cast<const uint8_t*>(p.A);
    const uint8_t* A_end = A8 + p.M * (int64_t)row_bytes;
    // MODE 3: the kept tiles first, in their stages
    const int first = MODE == 3 ? n - kept : 0;
    int b = first % NST, it = 0;
    uint32_t parity = (uint32_t)(first / NST) & 1u;
    for (int use = first; use < uses; ++use, ++it) {
        const int64_t m0 = tile_of(use) * TR;
        const int nr = p.M - m0 < TR ? (int)(p.M - m0) : TR;
        tc::wait_bounded(tc::smem_u32(&full_bar[b]), parity, abort_flag, p.timeout_ns, p.err, kErrWait);
        if (MODE == 2) consumer_sync();       // every consumer has waited: the abort test below is uniform
        if (tc::abort_raised(abort_flag)) break;
        const uint8_t* rows_b = rows_s + (size_t)(b * TR) * S;
        if (p.demote) {
            // the absmax pass kept these lines in L2 with priority; hand them back
            const uint8_t* lo = A8 + m0 * (int64_t)row_bytes;
            const uint8_t* hi = lo + (int64_t)nr * row_bytes;
            const uint8_t* l0 = reinterpret_cast<const uint8_t*>(((uintptr_t)lo + 127u) & ~(uintptr_t)127u);
            for (const uint8_t* l = l0 + 128 * tid; l < hi && l + 128 <= A_end; l += 128 * nthr_c)
                asm volatile("applypriority.global.L2::evict_normal [%0], 128;" ::"l"(l) : "memory");
        }
        GConst (*kc)[2] = kc_s[it & 1];
        if (MODE == 2) {
            if (warp < nr) {
                float f0, f1;
                row_group_max(rows_b + (size_t)warp * S, grp_s, K, f0, f1);
                if (lane == 0) {
                    p.s_a[(m0 + warp) * 2 + 0] = f0;
                    p.s_a[(m0 + warp) * 2 + 1] = f1;
                    kc[warp][0] = gconst(f0, p.g[0].bits_a);
                    kc[warp][1] = gconst(f1, p.g[1].bits_a);
                }
            }
            consumer_sync();
        }
        // ---- codes: lane per packed position; chunks of up to 8 blocks, rows inner ----
        const uint32_t rows_ba = fresh(rows_a + (uint32_t)(b * TR) * S);
        const uint32_t codes_a = tc::smem_u32(codes_s);
        for (int c = 0; c < nbw; c += 8) {
            const int nc = min(8, nbw - c);
            codes_chunk8<MODE>(rows_ba, codes_a, offs_s, gbase + (bw0 + c) * 32 + lane, nc, rr0, rgs, nr, S, npos, kc, kg,
                               g, lv, row_bytes);
        }
        __syncwarp();
        // this warp no longer reads the stage's rows
        if (lane == 0) tc::mbar_arrive(tc::smem_u32(&empty_bar[b]));
        // ---- pack: lane per (row, 32-code block): block lane % 8 of each chunk, rows lane / 8 and + 4 ----
        for (int c = 0; c < nbw; c += 8) {
            const int j = lane & 7;
            if (c + j < nbw) {
                const int kbg = bw0 + c + j;
#pragma unroll
                for (int h = 0; h < kGatherMaxRows / 4; ++h) {
                    const int r = rr0 + ((lane >> 3) + 4 * h) * rgs;
                    if (r < nr) {
                        const uint4* src = reinterpret_cast<const uint4*>(codes_s + (size_t)r * npos + gbase + kbg * 32);
                        const uint4 lo = src[0], hi = src[1];
                        const uint32_t ow[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                        store_block32_n(bits, ow, p.Ap + (m0 + r) * (int64_t)p.a_row_bytes + a_off + kbg * 4 * bits);
                    }
                }
            }
        }
        __syncwarp();   // the warp's codes are packed before the next tile overwrites them
        if (++b == NST) {
            b = 0;
            parity ^= 1u;
        }
    }
}

}  // namespace

namespace {

struct GatherPlan {
    int32_t tile_rows, stages, row_stride, npos;
    int32_t bpw, w0, wb, rg, nwc;
    size_t smem;
};

// mode as the kernel's MODE.
bool gather_plan(const LayoutGeom& geo, int mode, int64_t M, const void* A, GatherPlan* pl) {
    if (geo.K % 8 != 0 || (uintptr_t)A % 16 != 0) return false;
    const int nblk0 = geo.g[0].pa / 32, nblk1 = geo.g[1].pa / 32;
    if (nblk0 + nblk1 == 0) return false;
    pl->npos = geo.g[0].pa + geo.g[1].pa;
    pl->row_stride = ((2 * geo.K + 16) + 15) & ~15;
    // block ranges of 8 blocks (whole 8-wide chunks), or of a multiple of 8 where
    // the row needs more ranges than there are warps; warps left over split
    // the tile's rows
    for (pl->bpw = 8;; pl->bpw += 8) {
        pl->w0 = (nblk0 + pl->bpw - 1) / pl->bpw;
        pl->wb = pl->w0 + (nblk1 + pl->bpw - 1) / pl->bpw;
        if (pl->wb <= kGatherConsumerWarps) break;
    }
    pl->rg = kGatherConsumerWarps / pl->wb;
    const size_t budget = kGatherSmemBudget;
    const size_t fixed = (((size_t)pl->npos * (mode == 3 ? 2 : 4) + 15) & ~(size_t)15) +
                         (mode == 2 ? (((size_t)geo.K * 2 + 15) & ~(size_t)15) : 0) +
                         (mode == 3 ? (((size_t)geo.K / 8 + 19) & ~(size_t)15) : 0) + 16;
    if (fixed >= budget) return false;
    // a tile of up to eight rows per warp (MODE 2: eight in all) with as many stages as fit (at
    // least two, three for tiles of short rows), else fewer rows; then no more rows than an
    // SM's share needs in that many tiles, so that all SMs take the same number
    const size_t per_row = (size_t)pl->row_stride;
    const int64_t sms = num_sms() > 0 ? num_sms() : 1;
    auto stages_of = [&](int64_t t) {
        const size_t codes = ((size_t)t * pl->npos + 15) & ~(size_t)15;
        if (fixed + codes >= budget) return (int64_t)0;
        const int64_t n = (int64_t)((budget - fixed - codes) / (t * per_row));
        return n > kGatherMaxStages ? (int64_t)kGatherMaxStages : n;
    };
    int64_t tr = mode == 2 ? kGatherMaxRows : kGatherMaxRows * pl->rg;
    while (tr >= 1 && stages_of(tr) < (tr > kGatherMaxRows ? 3 : 2)) --tr;
    if (tr < 1) return false;
    const int64_t share = (M + sms - 1) / sms, rounds = (share + tr - 1) / tr;
    tr = (share + rounds - 1) / rounds;
    const int64_t nst = stages_of(tr);
    if (tr < 1) return false;
    pl->tile_rows = (int32_t)tr;
    pl->stages = (int32_t)nst;
    if (pl->rg > pl->tile_rows) pl->rg = pl->tile_rows;
    // exactly the warps that take blocks, and one per tile row at least (per-row maxima)
    pl->nwc = pl->wb * pl->rg < kGatherMinConsumerWarps ? kGatherMinConsumerWarps : pl->wb * pl->rg;
    pl->smem = fixed + (((size_t)tr * pl->npos + 15) & ~(size_t)15) + (size_t)nst * tr * per_row;
    return pl->smem <= budget;
}

int gather_mode(int32_t scale_mode) {
    return scale_mode == SONIQ_SCALE_CALIBRATED ? 0 : (scale_mode == SONIQ_SCALE_PER_ROW ? 2 : 1);
}

const void* gather_fn(int mode) {
    return mode == 0   ? (const void*)quantize_gather_kernel<0>
           : mode == 1 ? (const void*)quantize_gather_kernel<1>
           : mode == 2 ? (const void*)quantize_gather_kernel<2> : (const void*)quantize_gather_kernel<3>;
}

// Kernel parameters and attributes for a plan.
cudaError_t gather_setup(const LayoutGeom& geo, const GatherPlan& pl, int mode, const int32_t* perm, const uint16_t* A,
                         int64_t M, float* s_a, uint8_t* Ap, GatherParams* p) {
    p->A = A;
    p->Ap = Ap;
    p->s_a = s_a;
    p->perm = perm;
    p->err = device_error_word();
    if (p->err == nullptr) return cudaErrorNotSupported;
    p->timeout_ns = 2000000000LL;
    p->M = M;
    p->K = geo.K;
    p->a_row_bytes = geo.a_row_bytes;
    p->demote = 0;
    p->g[0] = geo.g[0];
    p->g[1] = geo.g[1];
    p->nblk0 = geo.g[0].pa / 32;
    p->nblk = p->nblk0 + geo.g[1].pa / 32;
    p->bpw = pl.bpw;
    p->w0 = pl.w0;
    p->wb = pl.wb;
    p->rg = pl.rg;
    p->nwc = pl.nwc;
    p->row_stride = pl.row_stride;
    p->tile_rows = pl.tile_rows;
    p->stages = pl.stages;
    p->bar = nullptr;
    p->part = nullptr;
    p->err_bit = 0u;
    p->drop_arrival = 0;
    static bool attr_done[64][4] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_done[dev][mode]) {
        cudaError_t e = cudaFuncSetAttribute(gather_fn(mode), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kGatherSmemBudget);
        if (e == cudaSuccess) e = prefer_max_shared(gather_fn(mode));
        if (e != cudaSuccess) return e;
        attr_done[dev][mode] = true;
    }
    return cudaSuccess;
}

}  // namespace

bool quantize_gather_supported(const LayoutGeom& geo, int32_t scale_mode, const void* A) {
    GatherPlan pl;
    return gather_plan(geo, gather_mode(scale_mode), (int64_t)1 << 31, A, &pl);
}

// Tiled quantize with bulk-staged rows (quantize_gather_kernel).  Needs rows
// of 16-byte-aligned 16-byte multiples (K % 8 == 0, A 16-byte aligned) and
// room for at least one row per stage; returns cudaErrorNotSupported
// otherwise.  scale_mode PER_ROW finds the scales; the others read s_a[2].
// demote: the input's L2 lines were read with an evict-last policy (the
// absmax pass), and their priority is reset as they are read here.
cudaError_t launch_quantize_gather(const LayoutGeom& geo, const int32_t* perm, const uint16_t* A, int64_t M,
                                   int32_t scale_mode, bool demote, float* s_a, uint8_t* Ap, cudaStream_t st) {
    const int mode = gather_mode(scale_mode);
    GatherPlan pl;
    if (M < 1 || !gather_plan(geo, mode, M, A, &pl)) return cudaErrorNotSupported;
    GatherParams p;
    cudaError_t e = gather_setup(geo, pl, mode, perm, A, M, s_a, Ap, &p);
    if (e != cudaSuccess) return e;
    p.demote = demote ? 1 : 0;
    const int64_t ntiles = (M + pl.tile_rows - 1) / pl.tile_rows, cap = num_sms();
    const dim3 grid((unsigned)(ntiles < cap ? ntiles : cap)), block((unsigned)(32 * (p.nwc + 1)));
    e = mode == 0   ? launch_pdl(quantize_gather_kernel<0>, grid, block, pl.smem, st, p)
        : mode == 1 ? launch_pdl(quantize_gather_kernel<1>, grid, block, pl.smem, st, p)
                    : launch_pdl(quantize_gather_kernel<2>, grid, block, pl.smem, st, p);
    if (e != cudaSuccess) return e;
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_quantize_stream(const LayoutGeom& geo, const int32_t* perm, const uint16_t* A, int64_t M, float* s_a,
                                   uint8_t* Ap, cudaStream_t st, unsigned* bar, float* part, int max_ctas,
                                   unsigned err_bit) {
    GatherPlan pl;
    if (M < 1 || bar == nullptr || part == nullptr || !gather_plan(geo, 3, M, A, &pl)) return cudaErrorNotSupported;
    GatherParams p;
    cudaError_t e = gather_setup(geo, pl, 3, perm, A, M, s_a, Ap, &p);
    if (e != cudaSuccess) return e;
    p.bar = bar;
    p.part = part;
    p.err_bit = err_bit;
    const int64_t ntiles = (M + pl.tile_rows - 1) / pl.tile_rows, cap = num_sms();
    const int64_t grid = ntiles < cap ? ntiles : cap;
    if (grid > max_ctas) return cudaErrorNotSupported;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)(32 * (p.nwc + 1)));
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    p.drop_arrival = take_drop_arrival() ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, quantize_gather_kernel<3>, p);
    if (e == cudaSuccess) note_launch();
    return e;
}

}  // namespace soniq

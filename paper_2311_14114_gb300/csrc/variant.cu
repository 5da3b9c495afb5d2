// Quantize and pack for the layout variants (linear layers):
//   * signed activations: Eq. (1) applied to the activation, codes in
//     [-2^(n-1), 2^(n-1) - 1] stored as n-bit two's complement (the
//     transformer-layer reading of Sec. 3);
//   * one-bit +-1 groups (Sec. 4.2, XNOR and POPCOUNT for one-bit channels):
//     code +1 for x >= 0 and -1 otherwise on both sides, stored as the bit
//     (code + 1) / 2;
//   * scale runs along K: a group's packed positions are cut into runs of
//     sub_k, each with its own max-abs scale (the fine scale groups of the
//     evaluation setup); scale arrays are [rows or 1][2][nb].
// Rows are staged whole in shared memory, several at a time (variant_rows_kernel);
// rows too long for that, and a few long rows under given scales, take two plain
// kernels that read through the permutation from global memory.
#include <cuda_fp16.h>
#include <stdint.h>

#include "soniq_device.cuh"
#include "soniq_internal.h"
#include "tc_ptx.cuh"

namespace soniq {
namespace {

constexpr int kAbsmaxThreads = 256;
constexpr int kMaxRuns = 512;   // 65536 / 128

template <typename T>
__device__ __forceinline__ float load_x(const T* X, int64_t i);
template <>
__device__ __forceinline__ float load_x<uint16_t>(const uint16_t* X, int64_t i) {
    return __half2float(__ushort_as_half(X[i]));
}
template <>
__device__ __forceinline__ float load_x<float>(const float* X, int64_t i) {
    return X[i];
}

struct VGeo {
    int32_t K, count0, count1, sub_k, nb;
    int32_t bits[2];
    int32_t kind[2];        // 0 unsigned, 1 signed (Eq. (1)), 2 +-1
    int32_t off[2];         // byte offset of group g in a packed row
    int32_t blocks[2];      // 32-code blocks of group g in a packed row
    int32_t row_bytes;
};

__device__ __forceinline__ int run_of(int j, int sub_k) { return sub_k > 0 ? j / sub_k : 0; }

// Max |x| per (group, run) of each row (per_row) or of all rows; s must be
// zero before a per-tensor launch (maxima are merged with atomicMax on the
// bit patterns, which order non-negative floats and infinity; NaN, whose
// patterns lie above infinity's, is skipped as the other max-abs passes skip it).
template <typename T>
__global__ void __launch_bounds__(kAbsmaxThreads) variant_absmax_kernel(const T* X, int64_t rows, const int32_t* perm,
                                                                        VGeo v, int per_row, float* s) {
    __shared__ unsigned smax[2 * kMaxRuns];
    const int nkeys = 2 * v.nb;
    for (int i = threadIdx.x; i < nkeys; i += blockDim.x) smax[i] = 0u;
    __syncthreads();
    for (int64_t m = blockIdx.x; m < rows; m += gridDim.x) {
        for (int p = threadIdx.x; p < v.K; p += blockDim.x) {
            const int g = p < v.count0 ? 0 : 1;
            const int j = g == 0 ? p : p - v.count0;
            const float a = fabsf(load_x<T>(X, m * v.K + perm[p]));
            if (a == a) atomicMax(&smax[g * v.nb + run_of(j, v.sub_k)], __float_as_uint(a));
        }
        if (per_row) {
            __syncthreads();
            for (int i = threadIdx.x; i < nkeys; i += blockDim.x) {
                s[m * nkeys + i] = __uint_as_float(smax[i]);
                smax[i] = 0u;
            }
            __syncthreads();
        }
    }
    if (!per_row) {
        __syncthreads();
        for (int i = threadIdx.x; i < nkeys; i += blockDim.x)
            if (smax[i] != 0u) atomicMax(reinterpret_cast<unsigned*>(s) + i, smax[i]);
    }
}

// One warp per (row, group, 32-code block): lane i takes code i of the block.
template <typename T>
__global__ void __launch_bounds__(256) variant_codes_kernel(const T* X, int64_t rows, const int32_t* perm, VGeo v,
                                                            const float* s, int per_row, int is_weight,
                                                            uint8_t* out) {
    const int lane = threadIdx.x & 31;
    const int64_t nblk = (int64_t)v.blocks[0] + v.blocks[1];
    const int64_t items = rows * nblk;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = warp0; it < items; it += nwarps) {
        const int64_t m = it / nblk;
        int blk = (int)(it - m * nblk);
        const int g = blk < v.blocks[0] ? 0 : 1;
        if (g == 1) blk -= v.blocks[0];
        const int n = v.bits[g];
        const int count = g == 0 ? v.count0 : v.count1;
        const int base = g == 0 ? 0 : v.count0;
        const int j = blk * 32 + lane;
        uint32_t pattern = 0u;
        if (j < count) {
            const float x = load_x<T>(X, m * v.K + perm[base + j]);
            const float sc = s[((per_row ? m : 0) * 2 + g) * v.nb + run_of(j, v.sub_k)];
            if (v.kind[g] == 2) {
                pattern = x >= 0.0f ? 1u : 0u;
            } else if (v.kind[g] == 1 || is_weight) {
                pattern = (uint32_t)weight_code(x, sc, (float)(1 << (n - 1))) & ((1u << n) - 1u);
            } else {
                pattern = act_code(x, sc, (float)((1 << n) - 1));
            }
        }
        const uint32_t word = pack_block_warp(pattern, n);
        if (lane < n)
            reinterpret_cast<uint32_t*>(out + m * v.row_bytes + v.off[g] + (int64_t)blk * 4 * n)[lane] = word;
    }
}

// ---- staged rows ---------------------------------------------------------------
//
// The plain kernels are bound by latency: a dependent global load per code, an
// atomic per element for the maxima, a warp-wide OR per packed word.  Here a CTA copies a
// tile of rows with one bulk copy, and a warp takes items of it: a chunk (four 32-code
// blocks, which share a scale, since runs are multiples of 128 codes) in some of the rows.
// Lane = position within a block, so the permutation is read once per item; a chunk's
// maximum is one warp reduction, merged in shared memory; the code bytes are packed a
// 32-code block per lane.  Items are chunks and not whole runs: a layout without runs has
// one run per group, and one or two of the 16 warps would walk all of it.  Tiles hold no
// more rows than give every SM two CTAs.  Signed 4/8 bits, per row, us with the plain
// kernels, a warp per run in tiles of eight rows, and now: without runs 16 x 4096 9.2, 119,
// 4.7; 8192 x 4096 347, 482, 67; weights 2048 x 4096 94, 243, 22; with 128-code runs
// 1001 x 3000 37.7, 13.7, 10.8.  Now bound by the codes' IEEE divisions and, at few rows, by a
// chain of an item's loads.
constexpr int kVarWarps = 16;
constexpr int kVarBlocks = 4;            // blocks of a chunk
constexpr int kVarRows = 8;              // rows of an item
constexpr size_t kVarSmem = 200 * 1024;
constexpr size_t kVarCodes = (size_t)kVarWarps * kVarRows * kVarBlocks * 32;   // the warps' code bytes
enum { VAR_GIVEN = 0, VAR_ROW = 1, VAR_MAX = 2 };   // scales given; found per row; per-tensor maxima only

template <typename T>
__device__ __forceinline__ float lds_x(const T* row, uint32_t c) {
    if constexpr (sizeof(T) == 2) return __half2float(__ushort_as_half(row[c]));
    else return row[c];
}

// An item's place: chunk c of group g (run b), its channels ch (-1: padding).
struct VItem {
    int g, c, b, ch[kVarBlocks];
    __device__ __forceinline__ VItem(const VGeo& v, const int32_t* perm, int chunk, int lane) {
        const int nc0 = v.blocks[0] / kVarBlocks;
        g = chunk >= nc0;
        c = chunk - (g ? nc0 : 0);
        b = v.sub_k > 0 ? c * (32 * kVarBlocks) / v.sub_k : 0;
        const int count = g ? v.count1 : v.count0, base = g ? v.count0 : 0;
#pragma unroll
        for (int j = 0; j < kVarBlocks; ++j) {
            const int pos = (c * kVarBlocks + j) * 32 + lane;
            ch[j] = pos < count ? __ldg(perm + base + pos) : -1;
        }
    }
};

// tile_rows rows per CTA, of which every split-th belongs to an item.
template <typename T, int MODE>
__global__ void __launch_bounds__(kVarWarps * 32) variant_rows_kernel(const T* X, int64_t rows, const int32_t* perm, VGeo v,
                                                                     float* s, int is_weight, int tile_rows, int split,
                                                                     uint8_t* out, unsigned* err, long long timeout_ns) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar_s;
    __shared__ uint32_t abort_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t m0 = (int64_t)blockIdx.x * tile_rows;
    const int nr = rows - m0 < tile_rows ? (int)(rows - m0) : tile_rows;
    const int nkeys = 2 * v.nb, items = (v.blocks[0] + v.blocks[1]) / kVarBlocks * split, nch = items / split;
    const uint32_t bar = tc::smem_u32(&bar_s), abort_flag = tc::smem_u32(&abort_s);
    // code bytes [warp][8 rows][4 blocks][32], the maxima [tile row][group][run] as bits, the rows
    uint8_t* codes = smem + (size_t)warp * (kVarRows * kVarBlocks * 32);
    uint32_t* max_s = reinterpret_cast<uint32_t*>(smem + kVarCodes);
    uint8_t* stage = smem + kVarCodes + (MODE == VAR_GIVEN ? 0 : ((size_t)tile_rows * nkeys * 4 + 15) / 16 * 16);
    if (threadIdx.x == 0) {
        tc::mbar_init(bar, 1);
        tc::set_flag(abort_flag, 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (MODE != VAR_GIVEN)
        for (int i = threadIdx.x; i < nr * nkeys; i += blockDim.x) max_s[i] = 0u;
    __syncthreads();
    tc::pdl_wait();      // launched with launch_pdl: every global access comes after this
    // The tile keeps its global address modulo 16: one bulk copy of the aligned interior,
    // plain loads of the few elements before and after it.
    const T* src = X + m0 * v.K;
    const uint32_t elems = (uint32_t)(nr * v.K);
    const uint32_t head = min(elems, (uint32_t)((16u - ((uintptr_t)src & 15u)) & 15u) / (uint32_t)sizeof(T));
    const uint32_t body = (elems - head) * (uint32_t)sizeof(T) & ~15u;
    T* rows_s = reinterpret_cast<T*>(stage + ((uintptr_t)src & 15u));
    if (threadIdx.x == 0) {
        tc::mbar_arrive_expect_tx(bar, body);
        if (body > 0) tc::bulk_load(tc::smem_u32(rows_s + head), src + head, body, bar);
    }
    if (threadIdx.x < head) rows_s[threadIdx.x] = src[threadIdx.x];
    for (uint32_t i = head + body / (uint32_t)sizeof(T) + threadIdx.x; i < elems; i += blockDim.x) rows_s[i] = src[i];
    __syncthreads();
    if (!tc::wait_bounded_warp(bar, 0u, abort_flag, timeout_ns, err, kErrWait)) {
        // the copy in flight lands before the CTA exits
        __shared__ uint32_t none_s;
        if (threadIdx.x == 0) {
            none_s = 0u;
            tc::wait_bounded(bar, 0u, tc::smem_u32(&none_s), timeout_ns, err, kErrWait);
        }
        tc::set_flag(abort_flag, 1);
    }

    if (MODE != VAR_GIVEN) {
        for (int it = warp; it < items; it += kVarWarps) {
            const int part = it / nch;
            const VItem w(v, perm, it - part * nch, lane);
            const int key = w.g * v.nb + w.b;
            for (int r = part; r < nr; r += split) {
                float m = 0.0f;
#pragma unroll
                for (int j = 0; j < kVarBlocks; ++j)
                    if (w.ch[j] >= 0) m = fmaxf(m, fabsf(lds_x<T>(rows_s + r * v.K, (uint32_t)w.ch[j])));   // skips NaN
                // non-negative floats order as their bits
                const uint32_t mb = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
                if (lane == 0) atomicMax(max_s + r * nkeys + key, mb);
            }
        }
    }
    __syncthreads();
    if (tc::abort_raised(abort_flag)) return;      // (a timed-out wait: nothing is written)
    if (MODE == VAR_MAX) {
        for (int key = threadIdx.x; key < nkeys; key += blockDim.x) {
            uint32_t m = 0u;
            for (int r = 0; r < nr; ++r) m = max(m, max_s[r * nkeys + key]);
            if (m != 0u) atomicMax(reinterpret_cast<unsigned*>(s) + key, m);
        }
        return;
    }
    if (MODE == VAR_ROW)
        for (int i = threadIdx.x; i < nr * nkeys; i += blockDim.x) s[m0 * nkeys + i] = __uint_as_float(max_s[i]);

    for (int it = warp; it < items; it += kVarWarps) {
        const int part = it / nch;
        const VItem w(v, perm, it - part * nch, lane);
        const int key = w.g * v.nb + w.b;
        // (selects, not indexed loads: an indexed parameter array would live in local memory)
        const int n = w.g ? v.bits[1] : v.bits[0], kind = w.g ? v.kind[1] : v.kind[0];
        const int off = w.g ? v.off[1] : v.off[0];
        const float half = (float)(1 << (n - 1)), levels = (float)((1 << n) - 1);
        const uint32_t mask = (1u << n) - 1u;
        float sc = MODE == VAR_GIVEN ? s[key] : 0.0f;
        int k = 0;                                 // rows of the item
        for (int r = part; r < nr; r += split, ++k) {
            if (MODE == VAR_ROW) sc = __uint_as_float(max_s[r * nkeys + key]);
#pragma unroll
            for (int j = 0; j < kVarBlocks; ++j) {
                uint32_t pattern = 0u;
                if (w.ch[j] >= 0) {
                    const float x = lds_x<T>(rows_s + r * v.K, (uint32_t)w.ch[j]);
                    if (kind == 2) pattern = x >= 0.0f ? 1u : 0u;
                    else if (kind == 1 || is_weight) pattern = (uint32_t)weight_code(x, sc, half) & mask;
                    else pattern = act_code(x, sc, levels);
                }
                codes[(k * kVarBlocks + j) * 32 + lane] = (uint8_t)pattern;
            }
        }
        __syncwarp();
        // lane -> (row, block)
        if (lane < k * kVarBlocks) {
            const int r = part + lane / kVarBlocks * split, j = lane % kVarBlocks;
            const uint4* c = reinterpret_cast<const uint4*>(codes + lane * 32);
            const uint4 lo = c[0], hi = c[1];
            const uint32_t o[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            store_block32_n(n, o, out + (m0 + r) * v.row_bytes + off + (int64_t)(w.c * kVarBlocks + j) * 4 * n);
        }
        __syncwarp();
    }
}
static_assert(kVarRows * kVarBlocks == 32, "an item's blocks are packed one per lane");

// Rows per tile of variant_rows_kernel, the rows' split and the shared memory; false where
// one row does not fit.
bool variant_plan(const VGeo& v, int64_t rows, size_t elem, int* tile_rows, int* split, size_t* smem) {
    const int nch = (v.blocks[0] + v.blocks[1]) / kVarBlocks;
    const size_t row = (size_t)v.K * elem + 2 * v.nb * 4;
    const size_t fixed = kVarCodes + 32;
    if (fixed + row > kVarSmem || nch == 0) return false;
    // rows of an item: up to eight; layouts with fewer chunks than warps split the tile's rows
    *split = nch < kVarWarps ? kVarWarps / nch : 1;
    int64_t tr = (int64_t)kVarRows * *split;
    // two CTAs per SM where that leaves two rows each, and as many tiles as CTAs fit
    const size_t half = kVarSmem / 2;
    const int64_t fit = (int64_t)(((fixed + 2 * row <= half ? half : kVarSmem) - fixed) / row);
    const int64_t ctas = 2 * (int64_t)num_sms(), share = (rows + ctas - 1) / ctas;
    if (tr > fit) tr = fit;
    if (tr > share) tr = share;
    if (*split > tr) *split = (int)tr;
    *tile_rows = (int)tr;
    *smem = kVarCodes + ((size_t)tr * 2 * v.nb * 4 + 15) / 16 * 16 + (size_t)tr * v.K * elem + 16;
    return (rows + tr - 1) / tr <= 2147483647;
}

template <typename T, int MODE>
cudaError_t launch_variant_rows(const T* X, int64_t rows, const int32_t* perm, const VGeo& v, float* s, int is_weight,
                                int tile_rows, int split, size_t smem, uint8_t* out, cudaStream_t st) {
    static bool attr_done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(variant_rows_kernel<T, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kVarSmem);
        if (e == cudaSuccess) e = prefer_max_shared((const void*)variant_rows_kernel<T, MODE>);
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
    unsigned* err = device_error_word();
    if (err == nullptr) return cudaErrorUnknown;
    const int64_t tiles = (rows + tile_rows - 1) / tile_rows;
    const cudaError_t e = launch_pdl(variant_rows_kernel<T, MODE>, dim3((unsigned)tiles), dim3(kVarWarps * 32), smem, st, X,
                                     rows, perm, v, s, is_weight, tile_rows, split, out, err, 2000000000LL);
    if (e == cudaSuccess) note_launch();
    return e;
}

VGeo make_vgeo(const LayoutGeom& geo, bool weight) {
    VGeo v{};
    v.K = geo.K;
    v.count0 = geo.g[0].count;
    v.count1 = geo.g[1].count;
    v.sub_k = geo.sub_k;
    v.nb = geo.nb;
    for (int g = 0; g < 2; ++g) {
        const GroupGeom& G = geo.g[g];
        v.bits[g] = weight ? G.bits_w : G.bits_a;
        v.kind[g] = weight ? (geo.act_kind[g] == 2 ? 2 : 1) : geo.act_kind[g];
        v.off[g] = weight ? G.w_off : G.a_off;
        v.blocks[g] = (weight ? G.pw : G.pa) / 32;
    }
    v.row_bytes = weight ? geo.w_row_bytes : geo.a_row_bytes;
    return v;
}

template <typename T>
cudaError_t run_variant(const LayoutGeom& geo, const int32_t* perm, const T* X, int64_t rows, bool weight,
                        int32_t scale_mode, float* s, uint8_t* out, cudaStream_t st) {
    const VGeo v = make_vgeo(geo, weight);
    const int per_row = scale_mode == SONIQ_SCALE_PER_ROW;
    cudaError_t e = cudaSuccess;
    size_t smem = 0;
    int tr = 0, split = 0;
    // Given scales, few long rows: a tile of one row keeps 16 warps busy for K / 2048 items each,
    // where the plain kernel spreads the row's blocks over the chip (signed 4/8 bits, us, plain and
    // staged: 16 x 4096 2.6, 3.7; 64 x 4096 4.0, 3.6; 64 x 16384 9.2, 10.3; 256 x 4096 9.2, 4.5).
    const bool plain = scale_mode == SONIQ_SCALE_CALIBRATED && rows <= 64 && v.K >= 2048;
    if (!plain && variant_plan(v, rows, sizeof(T), &tr, &split, &smem)) {
        if (per_row) return launch_variant_rows<T, VAR_ROW>(X, rows, perm, v, s, weight, tr, split, smem, out, st);
        if (scale_mode != SONIQ_SCALE_CALIBRATED) {
            if ((e = cudaMemsetAsync(s, 0, sizeof(float) * 2 * v.nb, st)) != cudaSuccess) return e;
            if ((e = launch_variant_rows<T, VAR_MAX>(X, rows, perm, v, s, weight, tr, split, smem, out, st)) != cudaSuccess)
                return e;
        }
        return launch_variant_rows<T, VAR_GIVEN>(X, rows, perm, v, s, weight, tr, split, smem, out, st);
    }
    if (scale_mode != SONIQ_SCALE_CALIBRATED) {
        if (!per_row && (e = cudaMemsetAsync(s, 0, sizeof(float) * 2 * v.nb, st)) != cudaSuccess) return e;
        const int64_t cap = (int64_t)num_sms() * 8;
        const int grid = (int)(rows < cap ? rows : cap);
        variant_absmax_kernel<T><<<grid, kAbsmaxThreads, 0, st>>>(X, rows, perm, v, per_row, s);
        note_launch();
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const int64_t items = rows * ((int64_t)v.blocks[0] + v.blocks[1]);
    const int64_t ctas = (items + 7) / 8;
    const int64_t cap = (int64_t)num_sms() * 16;
    variant_codes_kernel<T><<<(int)(ctas < cap ? ctas : cap), 256, 0, st>>>(X, rows, perm, v, s, per_row,
                                                                           weight ? 1 : 0, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_variant_quantize_act(const LayoutGeom& geo, const int32_t* perm, const uint16_t* A, int64_t M,
                                        int32_t scale_mode, float* s_a, uint8_t* Ap, cudaStream_t st) {
    return run_variant<uint16_t>(geo, perm, A, M, false, scale_mode, s_a, Ap, st);
}

cudaError_t launch_variant_pack_weights(const LayoutGeom& geo, const int32_t* perm, const float* W, int32_t N,
                                        float* s_w, uint8_t* Wp, cudaStream_t st) {
    return run_variant<float>(geo, perm, W, N, true, SONIQ_SCALE_PER_ROW, s_w, Wp, st);
}

}  // namespace soniq

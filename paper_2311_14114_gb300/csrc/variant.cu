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
// Rows are staged whole in shared memory, eight at a time (variant_rows_kernel);
// rows off the 16-byte grid, or too long for that, take two plain kernels that
// read through the permutation from global memory.
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
// atomic per element for the maxima, a warp-wide OR per packed word (14 us for the
// maxima and 24 us for the codes of a 1001 x 3000 fp16 input, 6 MB).  Here a CTA copies TR rows
// with one bulk copy, and a warp takes a run (the positions that share a scale) in all of
// them: lane = position within a 32-code block, so the permutation is read once per run;
// a row's maximum is one warp reduction, nothing is synchronised across warps, and the
// code bytes of the rows are packed a 32-code block per lane.
constexpr int kVarWarps = 16;
constexpr int kVarBlocks = 4;            // blocks of a run handled together
constexpr size_t kVarSmem = 200 * 1024;
enum { VAR_GIVEN = 0, VAR_ROW = 1, VAR_MAX = 2 };   // scales given; found per row; per-tensor maxima only

template <typename T>
__device__ __forceinline__ float lds_x(const T* row, uint32_t c) {
    if constexpr (sizeof(T) == 2) return __half2float(__ushort_as_half(row[c]));
    else return row[c];
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kVarWarps * 32) variant_rows_kernel(const T* X, int64_t rows, const int32_t* perm, VGeo v,
                                                                     float* s, int per_row, int is_weight, int tile_rows,
                                                                     uint8_t* out, unsigned* err, long long timeout_ns) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar_s;
    __shared__ uint32_t abort_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t m0 = (int64_t)blockIdx.x * tile_rows;
    const int nr = rows - m0 < tile_rows ? (int)(rows - m0) : tile_rows;
    const uint32_t bar = tc::smem_u32(&bar_s), abort_flag = tc::smem_u32(&abort_s);
    // code bytes [warp][tile row][4 blocks][32], then the rows
    uint8_t* codes = smem + (size_t)warp * tile_rows * kVarBlocks * 32;
    T* rows_s = reinterpret_cast<T*>(smem + (size_t)kVarWarps * tile_rows * kVarBlocks * 32);
    if (threadIdx.x == 0) {
        tc::mbar_init(bar, 1);
        tc::set_flag(abort_flag, 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    tc::pdl_wait();      // launched with launch_pdl: every global access comes after this
    const T* src = X + m0 * v.K;
    const int64_t elems = (int64_t)nr * v.K;
    const uint32_t bytes = (uint32_t)(elems * sizeof(T)), body = bytes & ~15u;
    if (threadIdx.x == 0) {
        tc::mbar_arrive_expect_tx(bar, body);
        if (body > 0) tc::bulk_load(tc::smem_u32(rows_s), src, body, bar);
    }
    for (int64_t i = body / sizeof(T) + threadIdx.x; i < elems; i += blockDim.x) rows_s[i] = src[i];   // a last tile's end
    __syncthreads();
    if (!tc::wait_bounded_warp(bar, 0u, abort_flag, timeout_ns, err, kErrWait)) {
        // the copy in flight lands before the CTA exits
        __shared__ uint32_t none_s;
        if (threadIdx.x == 0) {
            none_s = 0u;
            tc::wait_bounded(bar, 0u, tc::smem_u32(&none_s), timeout_ns, err, kErrWait);
        }
        return;
    }

    // a warp per key (group, run): its blocks kb0 .. kb1 - 1 of the group
    for (int key = warp; key < 2 * v.nb; key += kVarWarps) {
        const int g = key >= v.nb, b = key - (g ? v.nb : 0);
        const int rb = v.sub_k > 0 ? v.sub_k / 32 : v.blocks[g];
        const int kb0 = b * rb, kb1 = min(v.blocks[g], kb0 + rb);
        const int count = g ? v.count1 : v.count0, base = g ? v.count0 : 0;
        const int n = v.bits[g], kind = v.kind[g];
        const float half = (float)(1 << (n - 1)), levels = (float)((1 << n) - 1);
        const uint32_t mask = (1u << n) - 1u;
        // lane r: row r's scale
        float sc = 0.0f;
        if (MODE == VAR_GIVEN) {
            if (lane < nr) sc = s[((per_row ? m0 + lane : 0) * 2 + g) * v.nb + b];
        } else {
            for (int k = kb0; k < kb1; k += kVarBlocks) {
                int ch[kVarBlocks];
#pragma unroll
                for (int j = 0; j < kVarBlocks; ++j) {
                    const int pos = (k + j) * 32 + lane;
                    ch[j] = k + j < kb1 && pos < count ? __ldg(perm + base + pos) : -1;
                }
                for (int r = 0; r < nr; ++r) {
                    float m = 0.0f;
#pragma unroll
                    for (int j = 0; j < kVarBlocks; ++j)
                        if (ch[j] >= 0) m = fmaxf(m, fabsf(lds_x<T>(rows_s + (size_t)r * v.K, (uint32_t)ch[j])));   // skips NaN
                    // non-negative floats order as their bits
                    const uint32_t w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
                    if (lane == r) sc = fmaxf(sc, __uint_as_float(w));
                }
            }
            if (MODE == VAR_ROW && lane < nr) s[((m0 + lane) * 2 + g) * v.nb + b] = sc;
            if (MODE == VAR_MAX) {
                const uint32_t w = __reduce_max_sync(0xffffffffu, lane < nr ? __float_as_uint(sc) : 0u);
                if (lane == 0 && w != 0u) atomicMax(reinterpret_cast<unsigned*>(s) + key, w);
                continue;
            }
        }
        for (int k = kb0; k < kb1; k += kVarBlocks) {
            int ch[kVarBlocks];
#pragma unroll
            for (int j = 0; j < kVarBlocks; ++j) {
                const int pos = (k + j) * 32 + lane;
                ch[j] = k + j < kb1 && pos < count ? __ldg(perm + base + pos) : -1;
            }
            for (int r = 0; r < nr; ++r) {
                const float sr = __shfl_sync(0xffffffffu, sc, r);
#pragma unroll
                for (int j = 0; j < kVarBlocks; ++j) {
                    uint32_t pattern = 0u;
                    if (ch[j] >= 0) {
                        const float x = lds_x<T>(rows_s + (size_t)r * v.K, (uint32_t)ch[j]);
                        if (kind == 2) pattern = x >= 0.0f ? 1u : 0u;
                        else if (kind == 1 || is_weight) pattern = (uint32_t)weight_code(x, sr, half) & mask;
                        else pattern = act_code(x, sr, levels);
                    }
                    codes[(r * kVarBlocks + j) * 32 + lane] = (uint8_t)pattern;
                }
            }
            __syncwarp();
            // lane -> (row, block)
            for (int i = lane; i < nr * kVarBlocks; i += 32) {
                const int r = i / kVarBlocks, j = i % kVarBlocks;
                if (k + j < kb1) {
                    const uint4* c = reinterpret_cast<const uint4*>(codes + i * 32);
                    const uint4 lo = c[0], hi = c[1];
                    const uint32_t o[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                    store_block32_n(n, o, out + (m0 + r) * v.row_bytes + v.off[g] + (int64_t)(k + j) * 4 * n);
                }
            }
            __syncwarp();
        }
    }
}

// Rows per tile of variant_rows_kernel: the most of 8, 4, 2, 1 that fit and keep
// tiles on the 16-byte grid; 0: none.
template <typename T>
int variant_tile_rows(const T* X, int32_t K, size_t* smem) {
    for (int tr = 8; tr >= 1; tr /= 2) {
        const size_t row_bytes = (size_t)K * sizeof(T);
        *smem = (size_t)kVarWarps * tr * kVarBlocks * 32 + (size_t)tr * row_bytes;
        if ((uintptr_t)X % 16 == 0 && (tr * row_bytes) % 16 == 0 && *smem <= kVarSmem) return tr;
    }
    return 0;
}

template <typename T, int MODE>
cudaError_t launch_variant_rows(const T* X, int64_t rows, const int32_t* perm, const VGeo& v, float* s, int per_row,
                                int is_weight, int tile_rows, size_t smem, uint8_t* out, cudaStream_t st) {
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
                                     rows, perm, v, s, per_row, is_weight, tile_rows, out, err, 2000000000LL);
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
    const int tr = variant_tile_rows(X, v.K, &smem);
    if (tr > 0 && (rows + tr - 1) / tr <= 2147483647) {
        if (per_row)
            return launch_variant_rows<T, VAR_ROW>(X, rows, perm, v, s, 1, weight, tr, smem, out, st);
        if (scale_mode != SONIQ_SCALE_CALIBRATED) {
            if ((e = cudaMemsetAsync(s, 0, sizeof(float) * 2 * v.nb, st)) != cudaSuccess) return e;
            if ((e = launch_variant_rows<T, VAR_MAX>(X, rows, perm, v, s, 0, weight, tr, smem, out, st)) != cudaSuccess)
                return e;
        }
        return launch_variant_rows<T, VAR_GIVEN>(X, rows, perm, v, s, 0, weight, tr, smem, out, st);
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

// Mixed-precision GEMM for a few activation rows (decode batches, M <= 32) on
// warp-level tensor instructions: the exact integer GEMM of Sec. 3 / Sec. 4.2
// (Acc_g = sum over the channels of group g of u * j; Y = sum_g s_a s_w Acc_g /
// (L_w L_a)).
//
// What bounds it: the packed weight bytes, read once (20 MB for 11008 x 4096 at
// 3/6 bits, 3 us of HBM), as long as turning them into operands stays out of
// the way.  tcgen05 wants operands in shared memory, so the swap-AB kernel of
// skinny_gemm.cu writes every converted code there and fills 128 x 16 tiles from
// 86 CTAs: 33 us for 16 rows of that layer.  With mma.sync the operands are
// registers: a lane unpacks the words of its weight row's block straight into
// the B fragment, nothing converted is stored, and every SM takes a share of the
// rows.  The dot-product GEMV's work grows with M (16 us at M = 4); here it
// does not up to M = 16.
//
//   * Each CTA owns a contiguous range of weight rows and streams it through a
//     ring of 16-row stages (one bulk copy per row, a producer warp).
//   * The activation codes of all M rows sit in shared memory as bytes.
//   * 16 consumer warps split K: each takes a range of the 32-code blocks, for
//     every row of a stage.  Per block and eight weight rows: two m16n8k16 MMAs
//     (fp16 operands, fp32 accumulator).  The K order inside a block is the one
//     the packing gives: lane quarter q = lane % 4 holds codes 8 q .. 8 q + 7 of
//     both operands.
//   * Codes are integers up to 255 and -128: products and sums are exact in
//     fp32 while a warp's partial sum stays within 2^24; it is added to int32
//     totals in shared memory at least that often.
// Measured (11008 x 4096, 3/6 bits): 16.7 us at M = 16, 23 at M = 32; issue slots are
// half used, by unpacking and converting the weights.  Not faster: E4M3 MMAs
// (m16n8k32) for the low group, 17.0 us; activations kept as fp16 fragments, whose
// scattered writes cost more than the conversions saved, 29 us.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "packed_words.cuh"
#include "soniq_device.cuh"
#include "soniq_internal.h"
#include "tc_ptx.cuh"

namespace soniq {
namespace {

constexpr int kRowsWarps = 16;               // consumer warps
constexpr int kRowsThreads = (kRowsWarps + 1) * 32;
constexpr int kRowsTile = 16;                // weight rows per stage
constexpr int kRowsMaxStages = 8;
constexpr size_t kRowsSmem = 220 * 1024;

struct RowsParams {
    const uint8_t* Ap;
    const uint8_t* Wp;
    const float* s_a;
    const float* s_w;
    void* Y;
    int32_t* acc_dbg;
    unsigned* err;
    long long timeout_ns;
    int32_t M, N;
    int32_t a_row_bytes, w_row_bytes;
    int32_t s_a_per_row, out_bf16, drop_first;
    int32_t rows_cta;          // weight rows per CTA (a multiple of 16; the last CTA may have fewer)
    int32_t rows_pad;          // row stride of the totals
    int32_t acc_off, sw_off, act_off, buf_off;   // shared-memory offsets
    int32_t a_stride;          // bytes between the activation rows in shared memory
    int32_t wstride;           // bytes between the weight rows of a stage
    int32_t stages;
    int32_t nblk0, nblk;       // 32-code blocks of group 0 / of both groups
    int32_t seg_blocks[2];     // blocks a warp may sum in fp32
    GroupGeom g[2];
};

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four code bytes -> two fp16x2 words of (byte - off), bias = 1024 + off.
__device__ __forceinline__ void bytes_to_half(uint32_t x, __half2 bias, uint32_t& lo, uint32_t& hi) {
    bytes_to_magic_half2(x, lo, hi);
    lo = half2_sub(lo, bias);
    hi = half2_sub(hi, bias);
}

// Blocks kb0 .. kb1 - 1 of group g for the 16 weight rows staged at `rows`,
// added to the totals of rows r0 .. r0 + 15.
template <int N, int MT>
__device__ __forceinline__ void rows_blocks(const RowsParams& p, uint32_t rows, uint32_t act, int32_t* acc_s, int g,
                                            int kb0, int kb1, int r0) {
    const int lane = threadIdx.x & 31, row = lane >> 2, q = lane & 3;
    const __half2 bias_w = __half2half2(__ushort_as_half((unsigned short)(0x6400u + (1u << (N - 1)))));
    const __half2 bias_a = __half2half2(__ushort_as_half((unsigned short)0x6400u));
    const uint32_t flip = 0x01010101u << (N - 1);
    const bool vec8 = (p.g[g].w_off & 7) == 0;          // 16-byte-aligned rows; blocks of 4 N bytes, even N
    const uint32_t wsrc = rows + (uint32_t)(row * p.wstride + p.g[g].w_off);
    const uint32_t asrc = act + (uint32_t)(row * p.a_stride + (g ? p.nblk0 * 32 : 0) + 8 * q);
    for (int kb = kb0; kb < kb1;) {
        const int kend = min(kb1, kb + p.seg_blocks[g]);
        float acc[MT][2][4];
#pragma unroll
        for (int i = 0; i < MT * 8; ++i) (&acc[0][0][0])[i] = 0.0f;
#pragma unroll 2
        for (; kb < kend; ++kb) {
            // activation fragments of the block's two K steps
            uint32_t a[MT][2][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint2 x;
                    asm("ld.shared.v2.u32 {%0, %1}, [%2];"
                        : "=r"(x.x), "=r"(x.y)
                        : "r"(asrc + (uint32_t)((16 * mt + 8 * h) * p.a_stride + 32 * kb)));
                    bytes_to_half(x.x, bias_a, a[mt][0][h], a[mt][0][2 + h]);
                    bytes_to_half(x.y, bias_a, a[mt][1][h], a[mt][1][2 + h]);
                }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                PartWords<N, 4> w;
                w.load(SharedWords{wsrc + (uint32_t)(8 * nt * p.wstride + kb * 4 * N)}, q, N % 2 == 0 && vec8);
                uint32_t o[2], b[4];
                w.bytes(q, o);
                bytes_to_half(o[0] ^ flip, bias_w, b[0], b[1]);
                bytes_to_half(o[1] ^ flip, bias_w, b[2], b[3]);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_16816(acc[mt][nt], a[mt][0], b[0], b[1]);
                    mma_16816(acc[mt][nt], a[mt][1], b[2], b[3]);
                }
            }
        }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int m = 16 * mt + row + 8 * (e >> 1), n = r0 + 8 * nt + 2 * q + (e & 1);
                    if (m < p.M) atomicAdd(&acc_s[(g * p.M + m) * p.rows_pad + n], __float2int_rn(acc[mt][nt][e]));
                }
    }
}

template <int MT>
__global__ void __launch_bounds__(kRowsThreads, 1) rows_mma_kernel(const RowsParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full_bar[kRowsMaxStages], empty_bar[kRowsMaxStages];
    __shared__ uint32_t abort_s, none_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t abort_flag = tc::smem_u32(&abort_s);
    int32_t* acc_s = reinterpret_cast<int32_t*>(smem + p.acc_off);     // [2][M][rows_pad]
    float* sw_s = reinterpret_cast<float*>(smem + p.sw_off);           // [rows_cta][2]
    const uint32_t act = tc::smem_u32(smem + p.act_off), buf = tc::smem_u32(smem + p.buf_off);
    const uint32_t stage_bytes = (uint32_t)(kRowsTile * p.wstride);
    const int64_t n0 = (int64_t)blockIdx.x * p.rows_cta;
    const int nr = (int)(p.N - n0 < p.rows_cta ? p.N - n0 : p.rows_cta);
    const int tiles = (nr + kRowsTile - 1) / kRowsTile;
    if (tid == 0) {
        for (int i = 0; i < p.stages; ++i) {
            tc::mbar_init(tc::smem_u32(&full_bar[i]), 1);
            tc::mbar_init(tc::smem_u32(&empty_bar[i]), kRowsWarps);
        }
        tc::set_flag(abort_flag, 0);
        none_s = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 2 * p.M * p.rows_pad; i += kRowsThreads) acc_s[i] = 0;
    __syncthreads();
    tc::pdl_wait();      // launched with launch_pdl: every global access comes after this

    int b = 0;
    uint32_t ph = 0u;
    if (warp == kRowsWarps) {
        // ---- producer ----
        bool ok = true;
        int t = 0;
        for (; t < tiles; ++t) {
            if (t >= p.stages) {
                ok = tc::wait_bounded_warp(tc::smem_u32(&empty_bar[b]), ph ^ 1u, abort_flag, p.timeout_ns, p.err, kErrWait);
                if (!ok) break;
            }
            const int rows = nr - t * kRowsTile < kRowsTile ? nr - t * kRowsTile : kRowsTile;
            const uint32_t bar = tc::smem_u32(&full_bar[b]);
            if (!(p.drop_first && t == 0)) {
                if (lane == 0) tc::mbar_arrive_expect_tx(bar, (uint32_t)(rows * p.w_row_bytes));
                __syncwarp();
                if (lane < rows)
                    tc::bulk_load(buf + (uint32_t)b * stage_bytes + (uint32_t)(lane * p.wstride),
                                  p.Wp + (n0 + t * kRowsTile + lane) * p.w_row_bytes, (uint32_t)p.w_row_bytes, bar);
            }
            if (++b == p.stages) {
                b = 0;
                ph ^= 1u;
            }
        }
        // the copies in flight land before the CTA exits, also when it was abandoned
        if (lane == 0)
            for (int i = t > p.stages ? t - p.stages : 0; i < t; ++i)
                if (!(p.drop_first && i == 0))
                    tc::wait_bounded(tc::smem_u32(&full_bar[i % p.stages]), (uint32_t)(i / p.stages) & 1u,
                                     tc::smem_u32(&none_s), p.timeout_ns, p.err, kErrWait);
        return;
    }

    // ---- consumers: the activation rows as bytes, zero beyond PA up to the weights' PW ----
    for (int g = 0; g < 2; ++g) {
        const GroupGeom& G = p.g[g];
        const int nblk_a = G.pa / 32, nblk_w = G.pw / 32;
        uint8_t* dst = smem + p.act_off + (g ? p.nblk0 * 32 : 0);
        for (int item = tid; item < p.M * nblk_w; item += kRowsWarps * 32) {
            const int m = item / nblk_w, kb = item - m * nblk_w;
            uint32_t o[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
            if (kb < nblk_a) {
                const uint32_t* src =
                    reinterpret_cast<const uint32_t*>(p.Ap + (int64_t)m * p.a_row_bytes + G.a_off + kb * 4 * G.bits_a);
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) w[i] = i < G.bits_a ? __ldg(src + i) : 0u;
                block_to_bytes_n(G.bits_a, w, o);
            }
            uint4* d = reinterpret_cast<uint4*>(dst + m * p.a_stride + kb * 32);
            d[0] = make_uint4(o[0], o[1], o[2], o[3]);
            d[1] = make_uint4(o[4], o[5], o[6], o[7]);
        }
    }
    for (int i = tid; i < 2 * nr; i += kRowsWarps * 32) sw_s[i] = __ldg(p.s_w + n0 * 2 + i);
    asm volatile("bar.sync 1, %0;" ::"n"(kRowsWarps * 32) : "memory");
    uint32_t act_r = act;
    asm volatile("" : "+r"(act_r)::"memory");            // keeps the codes' loads behind the barrier

    const int b0 = (int)((int64_t)p.nblk * warp / kRowsWarps), b1 = (int)((int64_t)p.nblk * (warp + 1) / kRowsWarps);
    for (int t = 0; t < tiles; ++t) {
        if (!tc::wait_bounded_warp(tc::smem_u32(&full_bar[b]), ph, abort_flag, p.timeout_ns, p.err, kErrWait)) break;
        uint32_t rows = buf + (uint32_t)b * stage_bytes;
        asm volatile("" : "+r"(rows)::"memory");         // keeps the stage's loads behind the wait
#pragma unroll 1
        for (int g = 0; g < 2; ++g) {
            const int lo = g ? max(b0 - p.nblk0, 0) : min(b0, p.nblk0), hi = g ? b1 - p.nblk0 : min(b1, p.nblk0);
            if (lo >= hi) continue;
            const int r0 = t * kRowsTile;
            switch (p.g[g].bits_w) {
                case 1: rows_blocks<1, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                case 2: rows_blocks<2, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                case 3: rows_blocks<3, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                case 4: rows_blocks<4, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                case 5: rows_blocks<5, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                case 6: rows_blocks<6, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                case 7: rows_blocks<7, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
                default: rows_blocks<8, MT>(p, rows, act_r, acc_s, g, lo, hi, r0); break;
            }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(tc::smem_u32(&empty_bar[b]));
        if (++b == p.stages) {
            b = 0;
            ph ^= 1u;
        }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kRowsWarps * 32) : "memory");
    if (tc::abort_raised(abort_flag)) return;

    // ---- epilogue: thread per (activation row, weight row), weight rows fastest ----
    for (int i = tid; i < nr * p.M; i += kRowsWarps * 32) {
        const int m = i / nr, rr = i - m * nr;
        float y = 0.0f;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const GroupGeom& G = p.g[g];
            const int32_t a = acc_s[(g * p.M + m) * p.rows_pad + rr];
            if (p.acc_dbg != nullptr) p.acc_dbg[((int64_t)g * p.M + m) * p.N + n0 + rr] = a;
            if (G.pa == 0) continue;
            const float inv = 1.0f / ((float)((1 << G.bits_a) - 1) * (float)(1 << (G.bits_w - 1)));
            const float sw = sw_s[rr * 2 + g] * inv;
            const float sa = p.s_a_per_row ? __ldg(p.s_a + m * 2 + g) : __ldg(p.s_a + g);
            y = g == 0 ? (sa * sw) * (float)a : fmaf(sa * sw, (float)a, y);
        }
        const int64_t idx = (int64_t)m * p.N + n0 + rr;
        if (p.out_bf16) reinterpret_cast<__nv_bfloat16*>(p.Y)[idx] = __float2bfloat16_rn(y);
        else reinterpret_cast<__half*>(p.Y)[idx] = __float2half_rn(y);
    }
}

// Shared-memory layout; false if the activation rows and two stages do not fit.
bool rows_plan(const LayoutGeom& geo, int64_t M, int64_t N, RowsParams* p, size_t* smem) {
    if (M < 1 || M > 32 || N < 1 || geo.taps != 1 || geo.variant || geo.w_row_bytes % 16 != 0) return false;
    const int64_t codes = (int64_t)geo.g[0].pw + geo.g[1].pw;
    if (codes == 0) return false;
    const int64_t nsm = num_sms() > 0 ? num_sms() : 1, mt = M <= 16 ? 1 : 2;
    const int64_t tiles = (N + kRowsTile - 1) / kRowsTile, per = (tiles + nsm - 1) / nsm;
    p->rows_cta = (int32_t)(per * kRowsTile);
    p->rows_pad = (int32_t)((p->rows_cta + 31) / 32 * 32 + 8);      // lanes of one add on different banks
    p->nblk0 = geo.g[0].pw / 32;
    p->nblk = p->nblk0 + geo.g[1].pw / 32;
    p->a_stride = (int32_t)(codes + 32);                            // 8-byte reads of 4 rows on different banks
    int64_t ws = geo.w_row_bytes;
    if ((ws / 16) % 2 == 0) ws += 16;
    p->wstride = (int32_t)ws;
    int64_t o = 0;
    p->acc_off = (int32_t)o;
    o += 2 * M * p->rows_pad * 4;
    p->sw_off = (int32_t)o;
    o += (int64_t)p->rows_cta * 8;
    o = (o + 127) / 128 * 128;
    p->act_off = (int32_t)o;
    o += 16 * mt * (int64_t)p->a_stride;
    o = (o + 127) / 128 * 128;
    p->buf_off = (int32_t)o;
    const int64_t stage = kRowsTile * ws;
    int64_t st = ((int64_t)kRowsSmem - o) / stage;
    if (st < 2) return false;
    if (st > kRowsMaxStages) st = kRowsMaxStages;
    if (st > per) st = per;
    p->stages = (int32_t)st;
    *smem = (size_t)(o + st * stage);
    return true;
}

template <int MT>
cudaError_t run_rows(const RowsParams& p, size_t smem, cudaStream_t st) {
    static bool attr_done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(rows_mma_kernel<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kRowsSmem);
        if (e == cudaSuccess) e = prefer_max_shared((const void*)rows_mma_kernel<MT>);
        if (e != cudaSuccess) return e;
        attr_done[dev] = true;
    }
    const int64_t grid = (p.N + p.rows_cta - 1) / p.rows_cta;
    const cudaError_t e = launch_pdl(rows_mma_kernel<MT>, dim3((unsigned)grid), dim3(kRowsThreads), smem, st, p);
    if (e == cudaSuccess) note_launch();
    return e;
}

}  // namespace

bool rows_mma_supported(const LayoutGeom& geo, int64_t M, int64_t N) {
    RowsParams p;
    size_t smem;
    return rows_plan(geo, M, N, &p, &smem);
}

cudaError_t launch_rows_mma(const LayoutGeom& geo, const GemvArgs& a, bool drop_first, cudaStream_t st) {
    RowsParams p;
    size_t smem = 0;
    if (!rows_plan(geo, a.M, a.N, &p, &smem) || (uintptr_t)a.Wp % 16 != 0) return cudaErrorNotSupported;
    p.Ap = a.Ap;
    p.Wp = a.Wp;
    p.s_a = a.s_a;
    p.s_w = a.s_w;
    p.Y = a.Y;
    p.acc_dbg = a.acc_dbg;
    p.err = device_error_word();
    if (p.err == nullptr) return cudaErrorUnknown;
    p.timeout_ns = 2000000000LL;
    p.M = a.M;
    p.N = a.N;
    p.a_row_bytes = geo.a_row_bytes;
    p.w_row_bytes = geo.w_row_bytes;
    p.s_a_per_row = a.s_a_per_row;
    p.out_bf16 = a.out_bf16;
    p.drop_first = drop_first ? 1 : 0;
    for (int g = 0; g < 2; ++g) {
        p.g[g] = geo.g[g];
        const int64_t maxprod = (int64_t)((1 << geo.g[g].bits_a) - 1) << (geo.g[g].bits_w - 1);
        p.seg_blocks[g] = (int32_t)(((int64_t)1 << 24) / maxprod / 32);
    }
    return a.M <= 16 ? run_rows<1>(p, smem, st) : run_rows<2>(p, smem, st);
}

}  // namespace soniq

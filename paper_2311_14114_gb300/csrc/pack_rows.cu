// Weight quantize-and-pack with bulk-staged rows (Sec. 3 steps 1 and 3, Eq. (1)):
// per row and group s = max |w|, then the two's-complement codes of the row's
// packed positions.
//
// What bounds it: the fp32 rows are read once (4 bytes per weight against 0.4
// to 1 byte of codes written), so HBM is the floor.  Gathering every code's
// weight from global memory through the permutation instead is bound by the
// latency of those dependent loads: 274 us for 11008 x 4096 and 342 us for
// 4096 x 11008 (0.66 and 0.53 TB/s).
//
// How: persistent CTAs.  A producer warp keeps a ring of tiles of R whole rows
// in flight with one bulk copy per row; the consumer warps own fixed packed
// positions (lane = position within a 32-code block, VPT blocks of one group
// per warp), so the permutation is read once per CTA and lives in registers.
// A tile is gathered from shared memory into registers once; its maxima and
// its codes both come from those registers, and the stage is refilled
// meanwhile.  One CTA-wide barrier per tile combines the warps' maxima.  Codes
// leave as bytes through a per-warp buffer, from which each lane packs one
// 32-code block.  Measured: 11008 x 4096 in 45 us (4.0 TB/s), 4096 x 11008 in
// 55 us (3.3 TB/s); now bound by instruction issue and by the gathers' bank
// conflicts (1.9 wavefronts per load).
//
// Rows need not be 16-byte multiples: the copy takes the 16-byte-aligned
// interior, the producer's lanes move the (at most three) floats before and
// after it, and the row keeps its global address modulo 16 in its stage.
#include <stdint.h>

#include "soniq_device.cuh"
#include "soniq_internal.h"
#include "tc_ptx.cuh"

namespace soniq {
namespace {

constexpr int kPackMaxStages = 4;
constexpr size_t kPackSmemPerSm = 216 * 1024;

struct PackRowsParams {
    const float* W;
    uint8_t* Wp;
    float* s_w;
    const int32_t* perm;
    unsigned* err;
    long long timeout_ns;
    int32_t N, K, taps;
    int32_t L;               // floats per row: taps * K
    int32_t w_row_bytes;
    int32_t per_row;         // 0: the scales are s_w[0], s_w[1]
    int32_t stages, row_stride;   // tiles in the ring, bytes between staged rows
    int32_t zero_off;        // byte offset of a zero word behind a staged row
    int32_t w0, nwc;         // warps of group 0, consumer warps
    GroupGeom g[2];
};

__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ void sts_code(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

constexpr float kRound = 12582912.0f;              // 1.5 * 2^23
constexpr float kSafe = 0.5f - 8.0f * 0x1p-16f;    // distance to the nearest integer that decides the code

// Hands out a stage's address after its wait, which keeps the (movable) loads behind it.
__device__ __forceinline__ uint32_t after_wait(uint32_t v) {
    uint32_t r;
    asm volatile("mov.b32 %0, %1;" : "=r"(r) : "r"(v) : "memory");
    return r;
}

template <int VPT, int R, int WARPS, int CTAS>
__global__ void __launch_bounds__((WARPS + 1) * 32, CTAS) pack_rows_kernel(const PackRowsParams p) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full_bar[kPackMaxStages], empty_bar[kPackMaxStages];
    __shared__ uint32_t abort_s;
    // per tile: the rows' group maxima as bits [2][R] and, last, whether a wait ran out; the
    // third copy is cleared while the other two are in use
    __shared__ uint32_t red[3][2 * R + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t abort_flag = tc::smem_u32(&abort_s);
    uint8_t* rows_s = smem + ((size_t)p.nwc * VPT * R * 32 + 127) / 128 * 128;
    const uint32_t rows_a = tc::smem_u32(rows_s);
    const uint32_t stage_bytes = (uint32_t)(R * p.row_stride);
    const int64_t ntiles = ((int64_t)p.N + R - 1) / R;

    if (threadIdx.x == 0) {
        for (int b = 0; b < p.stages; ++b) {
            tc::mbar_init(tc::smem_u32(&full_bar[b]), 1);
            tc::mbar_init(tc::smem_u32(&empty_bar[b]), (uint32_t)p.nwc);
        }
        tc::set_flag(abort_flag, 0);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 3 * (2 * R + 1)) (&red[0][0])[threadIdx.x] = 0u;
    // a zero word behind every row, wherever the row starts within its first 16 bytes
    for (int i = threadIdx.x; i < 4 * R * p.stages; i += blockDim.x)
        *reinterpret_cast<float*>(rows_s + (size_t)(i >> 2) * p.row_stride + p.zero_off + 4 * (i & 3)) = 0.0f;
    __syncthreads();
    tc::pdl_wait();

    if (warp == p.nwc) {
        // ---- producer: R rows per stage ----
        int b = 0;
        uint32_t round = 0u;
        bool ok = true;
        for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
            if (round > 0u) {
                if (lane == 0)
                    ok = tc::wait_bounded(tc::smem_u32(&empty_bar[b]), (round - 1u) & 1u, abort_flag, p.timeout_ns,
                                          p.err, kErrWait);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (!ok) break;
                __syncwarp();
            }
            const uint32_t bar = tc::smem_u32(&full_bar[b]);
            const int nr = (int)(p.N - t * R < R ? p.N - t * R : R);
            for (int r = 0; r < nr; ++r) {
                const float* src = p.W + (t * R + r) * p.L;
                const int shift = (int)((uintptr_t)src & 15u);
                const uint32_t dst = rows_a + (uint32_t)b * stage_bytes + (uint32_t)(r * p.row_stride + shift);
                const int head = min(((16 - shift) & 15) / 4, p.L);      // floats before the aligned interior
                const int body = (p.L - head) & ~3;
                const int tail = p.L - head - body;
                if (lane == 0 && body > 0) {
                    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(4 * body)
                                 : "memory");
                    tc::bulk_load(dst + 4 * head, src + head, 4 * body, bar);
                }
                // lanes 0..2 the head, 4..6 the tail
                const int e = lane < 4 ? lane : head + body + lane - 4;
                if (lane < 4 ? lane < head : lane - 4 < tail)
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst + 4 * e), "f"(__ldg(src + e)) : "memory");
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(bar);
            if (++b == p.stages) {
                b = 0;
                ++round;
            }
        }
        if (lane == 0) {
            // the copies in flight land before the CTA exits, also when it was abandoned (the abort
            // flag may be up, so these waits get a flag of their own)
            __shared__ uint32_t none_s;
            none_s = 0u;
            for (int i = 0; i < p.stages; ++i) {
                const uint32_t uses = round + (i < b ? 1u : 0u);        // tiles the stage has taken
                if (uses > 0u)
                    tc::wait_bounded(tc::smem_u32(&full_bar[i]), (uses - 1u) & 1u, tc::smem_u32(&none_s), p.timeout_ns,
                                     p.err, kErrWait);
            }
        }
        return;
    }

    // ---- consumers: warp -> blocks bw0 .. bw0 + nbw - 1 of group g ----
    const int g = warp < p.w0 ? 0 : 1;
    const int bw0 = (g ? warp - p.w0 : warp) * VPT;
    const GroupGeom G = g ? p.g[1] : p.g[0];
    const int nbw = min(VPT, G.pw / 32 - bw0);
    const int bits = G.bits_w;
    const float half = (float)(1 << (bits - 1));
    const float kmax = kRound + (half - 1.0f);           // the largest code, rounded as below
    uint32_t off[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        off[i] = (uint32_t)p.zero_off;                   // padding and absent blocks: code 0
        if (i < nbw) {
            const int pos = (bw0 + i) * 32 + lane;
            const int t = p.taps == 1 ? 0 : pos / G.pa, c = pos - t * G.pa;
            if (t < p.taps && c < G.count) off[i] = 4u * (uint32_t)(t * p.K + __ldg(p.perm + G.perm_base + c));
        }
    }
    uint8_t* codes_s = smem + warp * VPT * R * 32;           // this warp's code bytes [R][VPT][32]
    const uint32_t codes_a = tc::smem_u32(codes_s) + (uint32_t)lane;
    const float t0 = p.per_row ? 0.0f : p.s_w[0], t1 = p.per_row ? 0.0f : p.s_w[1];
    uint8_t* out = p.Wp + G.w_off + (int64_t)bw0 * 4 * bits;

    int b = 0, par = 0;
    uint32_t parity = 0u;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t n0 = t * R;
        const int nr = (int)(p.N - n0 < R ? p.N - n0 : R);
        const bool ok = __all_sync(0xffffffffu, tc::wait_bounded(tc::smem_u32(&full_bar[b]), parity, abort_flag,
                                                                 p.timeout_ns, p.err, kErrWait));
        const uint32_t row0 = after_wait(rows_a + (uint32_t)b * stage_bytes);
        float v[R][VPT];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            // (rows past nr read an earlier tile's, and are not written)
            const uint32_t row = row0 + (uint32_t)(r * p.row_stride) + (uint32_t)((uintptr_t)(p.W + (n0 + r) * p.L) & 15u);
#pragma unroll
            for (int i = 0; i < VPT; ++i) v[r][i] = lds_f32(row + off[i]);
        }
        uint32_t mb[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float m = 0.0f;
#pragma unroll
            for (int i = 0; i < VPT; ++i) m = fmaxf(m, fabsf(v[r][i]));       // skips NaN, keeps infinities
            mb[r] = __reduce_max_sync(0xffffffffu, __float_as_uint(m));       // non-negative floats order as their bits
        }
        uint32_t* red_t = red[par];
        if (lane == 0) {
            tc::mbar_arrive(tc::smem_u32(&empty_bar[b]));              // the rows are in registers
#pragma unroll
            for (int r = 0; r < R; ++r) atomicMax(red_t + g * R + r, mb[r]);
            if (!ok) atomicOr(red_t + 2 * R, 1u);
        }
        par = par == 2 ? 0 : par + 1;
        if (threadIdx.x <= 2 * R) red[par][threadIdx.x] = 0u;          // last read two tiles ago
        asm volatile("bar.sync 1, %0;" ::"r"(32 * p.nwc) : "memory");
        if (red_t[2 * R] != 0u) break;                                 // every warp sees the same word
        if (threadIdx.x < 2 * R && (p.per_row || n0 > 0 || threadIdx.x >= 2)) {
            // scales, [row][group]; with given scales row 0 already holds them
            const int r = threadIdx.x >> 1, gg = threadIdx.x & 1;
            if (r < nr) p.s_w[(n0 + r) * 2 + gg] = p.per_row ? __uint_as_float(red_t[gg * R + r]) : (gg ? t1 : t0);
        }
        // lane r holds row r's scale and RN(1/s) * 2^(n-1)
        const float sl = !p.per_row ? (g ? t1 : t0) : lane < R ? __uint_as_float(red_t[g * R + lane]) : 0.0f;
        const float rl = sl > 0.0f ? __frcp_rn(sl) * half : 0.0f;
        // Eq. (1) from the estimate y = w * RN(1/s) * 2^(n-1), within a few ulps of 128 of
        // the IEEE quotient (under 3 even where 1/s is subnormal).  k = y + 1.5 * 2^23 rounds
        // y half to even into the low bits of k; a y within 8 ulps of 128 of a half-integer
        // (or NaN, or not finite because RN(1/s) * 2^(n-1) overflowed) redoes the IEEE division.
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float rh = __shfl_sync(0xffffffffu, rl, r);
            bool redo = false;
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const float y = __fmul_rn(v[r][i], rh);
                const float k = __fadd_rn(y, kRound);
                redo |= !(fabsf(__fsub_rn(y, __fsub_rn(k, kRound))) < kSafe);
                sts_code(codes_a + 32u * (r * VPT + i), __float_as_uint(fminf(k, kmax)));
            }
            if (__any_sync(0xffffffffu, redo)) {        // about one code in 2^12
                const float s = __shfl_sync(0xffffffffu, sl, r);
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const float y = __fmul_rn(v[r][i], rh);
                    if (!(fabsf(__fsub_rn(y, __fsub_rn(__fadd_rn(y, kRound), kRound))) < kSafe))
                        sts_code(codes_a + 32u * (r * VPT + i), (uint32_t)weight_code(v[r][i], s, half));
                }
            }
        }
        __syncwarp();
        // lane -> (row, 32-code block) of this warp; bits above the code width are masked by the packing
#pragma unroll
        for (int h = 0; h < (R * VPT + 31) / 32; ++h) {
            const int item = lane + 32 * h, r = item / VPT, i = item - r * VPT;
            if (r < nr && i < nbw) {
                const uint4* src = reinterpret_cast<const uint4*>(codes_s + item * 32);
                const uint4 lo = src[0], hi = src[1];
                const uint32_t o[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                store_block32_n(bits, o, out + (n0 + r) * p.w_row_bytes + i * 4 * bits);
            }
        }
        __syncwarp();      // the bytes are read before the next tile overwrites them
        if (++b == p.stages) {
            b = 0;
            parity ^= 1u;
        }
    }
}

template <int VPT, int R, int WARPS, int CTAS>
cudaError_t run_pack_rows(PackRowsParams& p, int nblk0, int nblk1, cudaStream_t st, bool* taken) {
    p.w0 = (nblk0 + VPT - 1) / VPT;
    p.nwc = p.w0 + (nblk1 + VPT - 1) / VPT;
    if (p.nwc > WARPS) return cudaSuccess;
    const size_t codes = ((size_t)p.nwc * VPT * R * 32 + 127) / 128 * 128;
    const int64_t stage = (int64_t)R * p.row_stride;
    const int64_t nst = ((int64_t)(kPackSmemPerSm / CTAS) - (int64_t)codes) / stage;
    if (nst < 2) return cudaSuccess;
    p.stages = (int32_t)(nst < kPackMaxStages ? nst : kPackMaxStages);
    *taken = true;
    const size_t smem = codes + (size_t)(p.stages * stage);
    const void* fn = (const void*)pack_rows_kernel<VPT, R, WARPS, CTAS>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kPackSmemPerSm / CTAS));
    if (e == cudaSuccess) e = prefer_max_shared(fn);
    if (e != cudaSuccess) return e;
    const int64_t cap = (int64_t)num_sms() * CTAS, ntiles = ((int64_t)p.N + R - 1) / R;
    e = launch_pdl(pack_rows_kernel<VPT, R, WARPS, CTAS>, dim3((unsigned)(ntiles < cap ? ntiles : cap)),
                   dim3((unsigned)(32 * (p.nwc + 1))), smem, st, p);
    if (e == cudaSuccess) note_launch();
    return e;
}

}  // namespace

cudaError_t launch_pack_rows(const LayoutGeom& geo, const int32_t* perm, const float* W, int32_t N, int32_t per_row,
                             uint8_t* Wp, float* s_w, cudaStream_t st) {
    const int64_t L = (int64_t)geo.taps * geo.K;
    const int nblk0 = geo.g[0].pw / 32, nblk1 = geo.g[1].pw / 32;
    if (L > 32768 || nblk0 + nblk1 == 0) return cudaErrorNotSupported;
    // A few short rows of one group are one warp's work either way, and staging them only adds to
    // it: a CTA per row of the plain kernel is as quick or quicker (us, plain and staged: 33 x 128
    // 2.7, 3.7; 162 x 128 2.9, 4.1; 162 x 79 2.9, 3.5; 645 x 128 3.1, 3.2; 2000 x 128 4.9, 3.3).
    if (nblk0 + nblk1 == 4 && L <= 128 && N <= 192) return cudaErrorNotSupported;
    PackRowsParams p;
    p.W = W;
    p.Wp = Wp;
    p.s_w = s_w;
    p.perm = perm;
    p.err = device_error_word();
    if (p.err == nullptr) return cudaErrorNotSupported;
    p.timeout_ns = 2000000000LL;
    p.N = N;
    p.K = geo.K;
    p.taps = geo.taps;
    p.L = (int32_t)L;
    p.w_row_bytes = geo.w_row_bytes;
    p.per_row = per_row;
    // the row at any offset below 16 bytes, then the zero word (at the same offset)
    p.zero_off = (int32_t)((4 * L + 15) / 16 * 16 + 16);
    p.row_stride = p.zero_off + 32;
    p.g[0] = geo.g[0];
    p.g[1] = geo.g[1];
    // Blocks per warp, rows per tile, warps, CTAs per SM: the narrowest rows that fit.  A warp
    // pays about 100 instructions per tile (wait, maxima, barrier, reciprocal, packing) next to
    // about 12 per 32 codes, so a tile of several rows shares them where the registers (rows x
    // blocks values and the offsets) allow.  11008 x 4096 at (8 blocks, R rows): R = 1 67 us,
    // R = 2 (two CTAs per SM) 52, R = 3 48, R = 4 45; 4096 x 11008: (16, 1) 55, (12, 2) 55 (spills),
    // (24, 2) 78; 3072 x 768: (4, 2) 6.9, (4, 4) 5.6.
    bool taken = false;
    cudaError_t e = run_pack_rows<4, 4, 8, 4>(p, nblk0, nblk1, st, &taken);
    if (!taken) e = run_pack_rows<8, 4, 17, 1>(p, nblk0, nblk1, st, &taken);
    if (!taken) e = run_pack_rows<16, 1, 23, 1>(p, nblk0, nblk1, st, &taken);
    if (!taken) e = run_pack_rows<24, 1, 23, 1>(p, nblk0, nblk1, st, &taken);
    return taken ? e : cudaErrorNotSupported;
}

}  // namespace soniq

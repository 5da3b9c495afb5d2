// Parts of a packed 32-code block: which words hold them, and their code bytes.
#pragma once

#include <stdint.h>

namespace soniq {

// The packed words that part `part` of PARTS equal parts of a block of N-bit
// codes needs (8 / PARTS output words of code bytes): its words of the 4- and
// 2-bit slices, the 1-bit slice's only word (N = 8: its own words).
template <int N, int PARTS>
struct PartWords {
    static constexpr int TW = 8 / PARTS;              // output words (four codes each)
    uint32_t w8[N == 8 ? TW : 1], w4[TW >= 2 ? TW / 2 : 1], w2[TW > 4 ? 2 : 1], w1;

    // from the block at src: src.one(i) is its word i, src.two(i) words i and i + 1
    // where vec8 (8-byte aligned)
    template <typename Src>
    __device__ __forceinline__ void load(const Src& src, int part, bool vec8) {
        if constexpr (N == 8) {
            pair_loads<TW>(src, part * TW, vec8, w8);
        } else {
            if constexpr ((N & 4) != 0) pair_loads<TW / 2>(src, part * (TW / 2), vec8, w4);
            constexpr int at2 = N & 4;
            if constexpr ((N & 2) != 0) {
                if constexpr (PARTS == 1) pair_loads<2>(src, at2, false, w2);
                else w2[0] = src.one(at2 + (PARTS == 2 ? part : part >> 1));
            }
            constexpr int at1 = (N & 4) + (N & 2);
            if constexpr ((N & 1) != 0) w1 = src.one(at1);
        }
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < (N == 8 ? TW : 1); ++i) w8[i] = 0u;
#pragma unroll
        for (int i = 0; i < (TW >= 2 ? TW / 2 : 1); ++i) w4[i] = 0u;
#pragma unroll
        for (int i = 0; i < (TW > 4 ? 2 : 1); ++i) w2[i] = 0u;
        w1 = 0u;
    }
    // byte b of o[k]: the pattern of code 4 (TW part + k) + b
    __device__ __forceinline__ void bytes(int part, uint32_t (&o)[TW]) const {
#pragma unroll
        for (int k = 0; k < TW; ++k) {
            if constexpr (N == 8) {
                o[k] = w8[k];
            } else {
                uint32_t v = 0u;
                if constexpr ((N & 4) != 0) v |= (w4[k >> 1] >> (4 * (k & 1))) & 0x0F0F0F0Fu;
                if constexpr ((N & 2) != 0) {
                    const uint32_t w = PARTS == 1 ? w2[k >> 2] : (PARTS == 2 ? w2[0] : w2[0] >> (4 * (part & 1)));
                    v |= ((w >> (2 * (k & 3))) & 0x03030303u) << (N & 4);
                }
                if constexpr ((N & 1) != 0)
                    v |= (((PARTS == 1 ? w1 : w1 >> (TW * part)) >> k) & 0x01010101u) << ((N & 4) + (N & 2));
                o[k] = v;
            }
        }
    }

private:
    template <int C, typename Src, int D>
    __device__ __forceinline__ static void pair_loads(const Src& src, int at, bool vec8, uint32_t (&w)[D]) {
        if constexpr (C % 2 == 0 && C > 0) {
            if (vec8) {
#pragma unroll
                for (int i = 0; i < C; i += 2) {
                    const uint2 v = src.two(at + i);
                    w[i] = v.x;
                    w[i + 1] = v.y;
                }
                return;
            }
        }
#pragma unroll
        for (int i = 0; i < C; ++i) w[i] = src.one(at + i);
    }
};

struct GlobalWords {
    const uint32_t* p;
    __device__ __forceinline__ explicit GlobalWords(const uint8_t* src) : p(reinterpret_cast<const uint32_t*>(src)) {}
    __device__ __forceinline__ uint32_t one(int i) const { return __ldg(p + i); }
    __device__ __forceinline__ uint2 two(int i) const { return __ldg(reinterpret_cast<const uint2*>(p + i)); }
};
struct SharedWords {
    uint32_t addr;
    __device__ __forceinline__ uint32_t one(int i) const {
        uint32_t v;
        asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr + 4u * (uint32_t)i));
        return v;
    }
    __device__ __forceinline__ uint2 two(int i) const {
        uint2 v;
        asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr + 4u * (uint32_t)i));
        return v;
    }
};

}  // namespace soniq

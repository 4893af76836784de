// Codes as packed 16-bit floats, for the kernels that multiply on warp-level 16-bit MMAs (split kernel, 16-bit form of the decode kernel).
#pragma once

#include "fbq_common.cuh"

namespace fbq {

// Codes become packed 16-bit floats with one LOP3 per pair ("bias-free" unpack): a field at bit p of a
// 16-bit half, OR-ed into the mantissa of MAGIC = 1024 (fp16) or 128 (bf16), is MAGIC + 2^p q.  Nothing is
// spent per element on removing MAGIC, 2^p or the zero point: x is staged divided by 2^p (in fp16 exact down to
// 2^(p - 14); the split kernel scales it up against that) and permuted into the order the unpacker produces,
// so the MMA yields sum x q + sum (MAGIC / 2^p) x; the second sum (P) and sum x (X0) depend on token and
// group only and are tabulated when x is staged, and a group contributes s (mma - P) - (s z) X0.
//   INT4: h[4i+e]  = codes (8i+e , 8i+e+4)  of word i          (i = 0..3, e = 0..3)
//   INT3: h[5i+f]  = codes (10i+f, 10i+5+f) of word i          (i = 0..2, f = 0..4);  h[15] = codes (30, 31)
__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t mask, uint32_t orv)
{
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(mask), "r"(orv));   // (a & mask) | orv
    return r;
}
template <int BITS, typename T> struct Unpack16;
template <> struct Unpack16<4, __half> {
    static constexpr float kMagic = 1024.f;
    static __device__ __forceinline__ constexpr int div_log2(int c) { return ((c & 7) & 1) ? 4 : 0; }   // odd nibbles sit 4 bits up
    static __device__ __forceinline__ void run(const uint32_t *w, uint32_t *h)
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t a = w[i], b = w[i] >> 8;
            h[4 * i + 0] = lop3_and_or(a, 0x000F000Fu, 0x64006400u);
            h[4 * i + 1] = lop3_and_or(a, 0x00F000F0u, 0x64006400u);
            h[4 * i + 2] = lop3_and_or(b, 0x000F000Fu, 0x64006400u);
            h[4 * i + 3] = lop3_and_or(b, 0x00F000F0u, 0x64006400u);
        }
    }
};
template <> struct Unpack16<4, __nv_bfloat16> {
    static constexpr float kMagic = 128.f;                     // 0x4300 | q is 128 + q in bf16 (7 mantissa bits)
    static __device__ __forceinline__ constexpr int div_log2(int) { return 0; }
    static __device__ __forceinline__ void run(const uint32_t *w, uint32_t *h)
    {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) h[4 * i + e] = lop3_and_or(w[i] >> (4 * e), 0x000F000Fu, 0x43004300u);
    }
};
template <> struct Unpack16<3, __half> {
    static constexpr float kMagic = 1024.f;
    static __device__ __forceinline__ constexpr int div_log2(int c)
    {
        if (c >= 30) return 0;
        const int f = (c % 10) % 5;                             // fields 0,3: bit 0; 1,4: bit 3; 2: bit 6 (3,4 after >> 9)
        return (f == 2) ? 6 : ((f == 1 || f == 4) ? 3 : 0);
    }
    static __device__ __forceinline__ void run(const uint32_t *w, uint32_t *h)
    {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint32_t a = w[i], b = w[i] >> 9;
            h[5 * i + 0] = lop3_and_or(a, 0x00070007u, 0x64006400u);
            h[5 * i + 1] = lop3_and_or(a, 0x00380038u, 0x64006400u);
            h[5 * i + 2] = lop3_and_or(a, 0x01C001C0u, 0x64006400u);
            h[5 * i + 3] = lop3_and_or(b, 0x00070007u, 0x64006400u);
            h[5 * i + 4] = lop3_and_or(b, 0x00380038u, 0x64006400u);
        }
        uint32_t l = lop3_and_or(w[0] >> 15, 0x00010001u, 0x64006400u);
        l = lop3_and_or(w[1] >> 14, 0x00020002u, l);
        h[15] = lop3_and_or(w[2] >> 13, 0x00040004u, l);
    }
};
template <> struct Unpack16<3, __nv_bfloat16> {
    static constexpr float kMagic = 128.f;
    static __device__ __forceinline__ constexpr int div_log2(int c)
    {
        if (c >= 30) return 0;
        const int f = (c % 10) % 5;                             // shifts 0, 6, 12: fields 0,2,4 at bit 0; 1,3 at bit 3
        return (f == 1 || f == 3) ? 3 : 0;
    }
    static __device__ __forceinline__ void run(const uint32_t *w, uint32_t *h)
    {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint32_t a = w[i], b = w[i] >> 6, c = w[i] >> 12;
            h[5 * i + 0] = lop3_and_or(a, 0x00070007u, 0x43004300u);
            h[5 * i + 1] = lop3_and_or(a, 0x00380038u, 0x43004300u);
            h[5 * i + 2] = lop3_and_or(b, 0x00070007u, 0x43004300u);
            h[5 * i + 3] = lop3_and_or(b, 0x00380038u, 0x43004300u);
            h[5 * i + 4] = lop3_and_or(c, 0x00070007u, 0x43004300u);
        }
        uint32_t l = lop3_and_or(w[0] >> 15, 0x00010001u, 0x43004300u);
        l = lop3_and_or(w[1] >> 14, 0x00020002u, l);
        h[15] = lop3_and_or(w[2] >> 13, 0x00040004u, l);
    }
};
// Position of code c (0..31) of a lane's 32-code run in that order: 2 * h_index + (0 = low half, 1 = high half).
template <int BITS> __device__ __forceinline__ int frag_pos(int c)
{
    if (BITS == 4) {
        const int i = c >> 3, e8 = c & 7;
        return 2 * (4 * i + (e8 & 3)) + (e8 >> 2);
    }
    if (c >= 30) return 2 * 15 + (c - 30);
    const int i = c / 10, f = c - 10 * i;
    return (f < 5) ? 2 * (5 * i + f) : 2 * (5 * i + f - 5) + 1;
}

}  // namespace fbq

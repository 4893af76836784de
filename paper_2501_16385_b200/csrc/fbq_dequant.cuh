// Packed codes to the activation type: s * (q - z) with one rounding, 32 codes at a time, in natural k order.
#pragma once

#include "fbq_common.cuh"

namespace fbq {

__device__ __forceinline__ uint32_t pf_lop3(uint32_t a, uint32_t mask, uint32_t orv)
{
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(mask), "r"(orv));   // (a & mask) | orv
    return r;
}
__device__ __forceinline__ uint32_t pf_prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Packed-pair arithmetic of the activation type on raw 32-bit registers.
template <typename T> struct P2;
template <> struct P2<__half> {
    static constexpr uint32_t kFmt = 0;              // instruction-descriptor format code
    static __device__ __forceinline__ uint32_t sub(uint32_t a, uint32_t b)
    {
        uint32_t r;
        asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    }
    static __device__ __forceinline__ uint32_t mul(uint32_t a, uint32_t b)
    {
        uint32_t r;
        asm("mul.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    }
    static __device__ __forceinline__ uint32_t fma(uint32_t a, uint32_t b, uint32_t c)
    {
        uint32_t r;
        asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
        return r;
    }
    static __device__ __forceinline__ uint32_t splat(float v)
    {
        __half2 h = __float2half2_rn(v);
        return *reinterpret_cast<uint32_t *>(&h);
    }
    static __device__ __forceinline__ uint32_t pack(float lo, float hi)
    {
        __half2 h = __floats2half2_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    }
};
template <> struct P2<__nv_bfloat16> {
    static constexpr uint32_t kFmt = 1;
    static __device__ __forceinline__ uint32_t sub(uint32_t a, uint32_t b)
    {
        uint32_t r;
        asm("sub.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    }
    static __device__ __forceinline__ uint32_t mul(uint32_t a, uint32_t b)
    {
        uint32_t r;
        asm("mul.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    }
    static __device__ __forceinline__ uint32_t fma(uint32_t a, uint32_t b, uint32_t c)
    {
        uint32_t r;
        asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
        return r;
    }
    static __device__ __forceinline__ uint32_t splat(float v)
    {
        __nv_bfloat162 h = __float2bfloat162_rn(v);
        return *reinterpret_cast<uint32_t *>(&h);
    }
    static __device__ __forceinline__ uint32_t pack(float lo, float hi)
    {
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    }
};

// Order of the 32 element pairs of one 64-wide K block as the dequantiser emits them
// (pair p occupies 32-bit word p of the block's shared-memory row).
template <int BITS> __device__ __forceinline__ constexpr int pair_lo(int p)
{
    if (BITS == 4) return 8 * (p / 4) + (p % 4);                       // word p/4: codes (e, e+4)
    const int r = p / 16, q = p % 16;                                  // run r of 32 codes
    return 32 * r + (q == 15 ? 30 : 10 * (q / 5) + (q % 5));
}
template <int BITS> __device__ __forceinline__ constexpr int pair_hi(int p)
{
    if (BITS == 4) return pair_lo<4>(p) + 4;
    const int r = p / 16, q = p % 16;
    return 32 * r + (q == 15 ? 31 : 10 * (q / 5) + 5 + (q % 5));
}

// s*(q - z) for 32 consecutive codes of one weight row (half a K block), as 16 packed pairs
// in the order above.  q - z is exact (exponent trick, integer-valued z); the product is
// rounded once to the activation type.  w: 4 words (INT4) or one run of 3 words (INT3).
template <int BITS, typename T> struct Dequant;
template <> struct Dequant<4, __half> {
    static __device__ __forceinline__ void run(const uint32_t *w, float s, float z, uint32_t *out)
    {
        const uint32_t c0 = P2<__half>::splat(1024.f + z), c1 = P2<__half>::splat(-(64.f + z)), s2 = P2<__half>::splat(s);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t a = w[i], b = w[i] >> 8;
            out[4 * i + 0] = P2<__half>::mul(P2<__half>::sub(pf_lop3(a, 0x000F000Fu, 0x64006400u), c0), s2);
            out[4 * i + 1] = P2<__half>::mul(P2<__half>::fma(pf_lop3(a, 0x00F000F0u, 0x64006400u), 0x2C002C00u, c1), s2);
            out[4 * i + 2] = P2<__half>::mul(P2<__half>::sub(pf_lop3(b, 0x000F000Fu, 0x64006400u), c0), s2);
            out[4 * i + 3] = P2<__half>::mul(P2<__half>::fma(pf_lop3(b, 0x00F000F0u, 0x64006400u), 0x2C002C00u, c1), s2);
        }
    }
};
template <> struct Dequant<4, __nv_bfloat16> {
    static __device__ __forceinline__ void run(const uint32_t *w, float s, float z, uint32_t *out)
    {
        using P = P2<__nv_bfloat16>;
        const uint32_t c0 = P::splat(128.f + z), s2 = P::splat(s);   // 0x4300 | q is 128 + q in bf16
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                out[4 * i + e] = P::mul(P::sub(pf_lop3(w[i] >> (4 * e), 0x000F000Fu, 0x43004300u), c0), s2);
    }
};
template <> struct Dequant<3, __half> {
    static __device__ __forceinline__ void run(const uint32_t *w, float s, float z, uint32_t *out)
    {
        using P = P2<__half>;
        const uint32_t c0 = P::splat(1024.f + z), n1 = P::splat(-(128.f + z)), n2 = P::splat(-(16.f + z)), s2 = P::splat(s);
        {
            const uint32_t *v = w;
            uint32_t *o = out;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const uint32_t a = v[i], b = v[i] >> 9;
                o[5 * i + 0] = P::mul(P::sub(pf_lop3(a, 0x00070007u, 0x64006400u), c0), s2);
                o[5 * i + 1] = P::mul(P::fma(pf_lop3(a, 0x00380038u, 0x64006400u), 0x30003000u, n1), s2);
                o[5 * i + 2] = P::mul(P::fma(pf_lop3(a, 0x01C001C0u, 0x64006400u), 0x24002400u, n2), s2);
                o[5 * i + 3] = P::mul(P::sub(pf_lop3(b, 0x00070007u, 0x64006400u), c0), s2);
                o[5 * i + 4] = P::mul(P::fma(pf_lop3(b, 0x00380038u, 0x64006400u), 0x30003000u, n1), s2);
            }
            uint32_t l = pf_lop3(v[0] >> 15, 0x00010001u, 0x64006400u);
            l = pf_lop3(v[1] >> 14, 0x00020002u, l);
            l = pf_lop3(v[2] >> 13, 0x00040004u, l);
            o[15] = P::mul(P::sub(l, c0), s2);
        }
    }
};
template <> struct Dequant<3, __nv_bfloat16> {
    static __device__ __forceinline__ void run(const uint32_t *w, float s, float z, uint32_t *out)
    {
        using P = P2<__nv_bfloat16>;
        const uint32_t c0 = P::splat(128.f + z), n1 = P::splat(-(16.f + z)), s2 = P::splat(s);
        {
            const uint32_t *v = w;
            uint32_t *o = out;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const uint32_t a = v[i], b = v[i] >> 6, c = v[i] >> 12;
                o[5 * i + 0] = P::mul(P::sub(pf_lop3(a, 0x00070007u, 0x43004300u), c0), s2);
                o[5 * i + 1] = P::mul(P::fma(pf_lop3(a, 0x00380038u, 0x43004300u), 0x3E003E00u, n1), s2);
                o[5 * i + 2] = P::mul(P::sub(pf_lop3(b, 0x00070007u, 0x43004300u), c0), s2);
                o[5 * i + 3] = P::mul(P::fma(pf_lop3(b, 0x00380038u, 0x43004300u), 0x3E003E00u, n1), s2);
                o[5 * i + 4] = P::mul(P::sub(pf_lop3(c, 0x00070007u, 0x43004300u), c0), s2);
            }
            uint32_t l = pf_lop3(v[0] >> 15, 0x00010001u, 0x43004300u);
            l = pf_lop3(v[1] >> 14, 0x00020002u, l);
            l = pf_lop3(v[2] >> 13, 0x00040004u, l);
            o[15] = P::mul(P::sub(l, c0), s2);
        }
    }
};

// Where Dequant leaves element e (0..31, natural k order) of its 32 codes: register and half.
template <int BITS> __device__ __forceinline__ constexpr int elem_reg(int e)
{
    if (BITS == 4) return 4 * (e / 8) + (e % 4);                       // word e/8: pairs (j, j+4)
    const int r = e / 32, q = e % 32;                                  // run r of 32 codes
    return 16 * r + (q >= 30 ? 15 : 5 * (q / 10) + (q % 10) % 5);
}
template <int BITS> __device__ __forceinline__ constexpr int elem_half(int e)
{
    if (BITS == 4) return (e % 8) / 4;
    const int q = e % 32;
    return q >= 30 ? q - 30 : (q % 10) / 5;
}
// Re-pair the 32 dequantised values into natural order: word p = elements (2p, 2p+1).
template <int BITS> __device__ __forceinline__ void natural_pairs(const uint32_t *d /*16*/, uint32_t *out /*16*/)
{
#pragma unroll
    for (int p = 0; p < 16; ++p) {
        const int a = elem_reg<BITS>(2 * p), ha = elem_half<BITS>(2 * p);
        const int b = elem_reg<BITS>(2 * p + 1), hb = elem_half<BITS>(2 * p + 1);
        out[p] = pf_prmt(d[a], d[b], (hb ? 0x7600u : 0x5400u) | (ha ? 0x32u : 0x10u));
    }
}

template <typename T> __device__ __forceinline__ unsigned short to_bits16(float v)
{
    return (unsigned short)(P2<T>::pack(v, 0.f) & 0xFFFFu);
}

}  // namespace fbq

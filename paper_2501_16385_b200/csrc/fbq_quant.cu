// Feedback quantiser (Section 4.1 of the paper): the main path of FBQuant stores
// Q(W - Sigma), Sigma = B.A, so that  W_F = Q(W - Sigma) + Sigma  stays within s/2 of W
// for a round-to-nearest quantiser (Eq. "diff" and the bound below it).  This is the
// offline step that produces the (codes, s, z) the inference kernels consume.
//
// Reading of "linear quantizer, group size 128, round to nearest with scaling factor s":
// asymmetric min-max per group of `group` consecutive input channels of one output row,
//     r = W - B.A                       s = max((max r - min r)/(2^bits - 1), 2^-14)
//     z = rint(-min r / s)              q = clamp(rint(r/s + z), 0, 2^bits - 1)   (ties to even)
// (constant group c: s = max(|c|, 2^-14), z = 1 if c < 0 else 0), with s and z rounded to
// fp16 first and the STORED values used for the codes, so that dequantisation inverts
// exactly what was coded.  Every rounding decision is taken in IEEE single precision with
// one operation per step (explicit _rn intrinsics: no contraction, no fast division), in
// the order the definition states, so that a CPU check can reproduce the codes bit for bit.
//
// Groups of 128 (the paper's): quantise_tile_kernel, 128 rows x one group per CTA, Sigma as a register-tiled
// product.  Other group sizes: quantize_feedback_kernel, one CTA per (group, row), a thread owns one k.
#include <cstring>

#include "fbq_common.cuh"
#include "fbq_ptx.cuh"

namespace fbq {
namespace {

template <typename T> __device__ __forceinline__ float ab_to_float(T v) { return ActTraits<T>::to_float(v); }
template <> __device__ __forceinline__ float ab_to_float<float>(float v) { return v; }

// (s, z) of a group from its extremes, as they are stored.
__device__ __forceinline__ void scale_and_zero(float mn, float mx, int bits, __half &s_h, __half &z_h)
{
    const float maxq = (float)((1 << bits) - 1), smin = 6.103515625e-05f;   // 2^-14
    float s, z;
    if (mx > mn) {
        s = fmaxf(__fdiv_rn(__fsub_rn(mx, mn), maxq), smin);
        const float sh = __half2float(__float2half_rn(s));
        z = rintf(__fdiv_rn(-mn, sh));
    } else {
        s = fmaxf(fabsf(mn), smin);
        z = (mn < 0.f) ? 1.f : 0.f;
    }
    s_h = __float2half_rn(s);
    z_h = __float2half_rn(z);
}

// codes, scales/zeros, WF and Delta (= W - W_F, the Delta_F of Section 4.2) are each optional.
template <typename T>
__global__ void quantize_feedback_kernel(const float *__restrict__ W, const T *__restrict__ A, const T *__restrict__ B,
                                         uint8_t *__restrict__ codes, __half *__restrict__ scales,
                                         __half *__restrict__ zeros, float *__restrict__ WF, float *__restrict__ Delta,
                                         int N, int K, int group, int bits, int rank)
{
    __shared__ float s_min[32], s_max[32];
    __shared__ float s_sz[2];
    const int n = blockIdx.x, g = blockIdx.y, i = threadIdx.x;     // rows vary fastest: neighbours share A's columns in L2
    const int G = K / group;
    const bool active = i < group;
    const int k = g * group + (active ? i : 0);
    float sigma = 0.f, r = 0.f;
    if (active) {
        for (int j = 0; j < rank; ++j)
            sigma = __fmaf_rn(ab_to_float<T>(B[(size_t)n * rank + j]), ab_to_float<T>(A[(size_t)j * K + k]), sigma);
        r = __fsub_rn(W[(size_t)n * K + k], sigma);
    }
    float mn = active ? r : INFINITY, mx = active ? r : -INFINITY;
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((i & 31) == 0) {
        s_min[i >> 5] = mn;
        s_max[i >> 5] = mx;
    }
    __syncthreads();
    if (i == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int w = 1; w < nw; ++w) {
            mn = fminf(mn, s_min[w]);
            mx = fmaxf(mx, s_max[w]);
        }
        __half s_h, z_h;
        scale_and_zero(mn, mx, bits, s_h, z_h);
        if (scales) {
            scales[(size_t)n * G + g] = s_h;
            zeros[(size_t)n * G + g] = z_h;
        }
        s_sz[0] = __half2float(s_h);
        s_sz[1] = __half2float(z_h);
    }
    __syncthreads();
    if (active) {
        const float sh = s_sz[0], zh = s_sz[1], maxq = (float)((1 << bits) - 1);
        float q = rintf(__fadd_rn(__fdiv_rn(r, sh), zh));
        q = fminf(fmaxf(q, 0.f), maxq);
        if (codes) codes[(size_t)n * K + k] = (uint8_t)q;
        const float wf = __fadd_rn(__fmul_rn(sh, __fsub_rn(q, zh)), sigma);
        if (WF) WF[(size_t)n * K + k] = wf;
        if (Delta) Delta[(size_t)n * K + k] = __fsub_rn(W[(size_t)n * K + k], wf);
    }
}

// 128 rows x one group of 128 per CTA.  What bounds it is Sigma: rank fused multiply-adds per weight, in index order
// (every rounding is part of the definition, so no tensor core): 11008 x 4096 at rank 64 is 2.9 G of them, beside 225 MB
// of W and codes (35 us).  A warp owns 16 rows x 128 k, a lane 4 k of each row, two rows per packed fma (fma.rn.f32x2: two
// IEEE fmas in one issue slot, at the rate of two single ones: 80 us here).  Shared memory is the other bound: per rank
// index a warp reads its 128 values of A (fp32, 4 wavefronts) and 16 of B (rows side by side, every lane the same: 8)
// for 16 cycles of multiply-adds.  (B as pairs (b, b) for two k per fma took 28 wavefronts: 160 us per 64 rank indices.)  32 rank indices are staged at a time, the next ones on their
// way to registers meanwhile.  The CTA's tile of W is requested first (cp.async, every thread its own 64 values) and is
// there when Sigma is.  Minimum and maximum of the 16 rows are 16 shuffles each (every step halves the rows a lane still
// carries) and leave a row to each pair of lanes, which fixes its (s, z).  The codes come from a product with 1/s and
// are taken only where they cannot depend on its error (codes_of_row): IEEE divisions one after another were a third of
// the kernel.  4096 x 11008, rank 64, INT3: 1009 us with a CTA per row and group, 177 us now (62 at rank 0).
constexpr int kQT = 128;                      // group size and rows of a tile
constexpr int kQJ = 32;                       // rank indices staged at a time
constexpr int kQThreads = 256;
constexpr size_t kQSmemW = (size_t)kQT * kQT * 4, kQSmemA = (size_t)kQJ * kQT * 4, kQSmemB = (size_t)kQJ * kQT * 4,
                 kQSmem = kQSmemW + kQSmemA + kQSmemB;          // 96 KB: two CTAs per SM

__device__ __forceinline__ void fma2(unsigned long long &d, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long twice(float v)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
struct alignas(16) Pair2 {
    unsigned long long x, y;
};

// Four codes q = clamp(rint(fl(fl(r / s) + z))) of one row.  r * (1/s) is within 3 ulp of fl(r / s); unless that error
// (and the rounding of the sum) could carry the sum across a rounding boundary, rint gives the same integer, and
// only then is the division done as the definition has it.  rint is an addition here (the sum is clamped first, so it
// fits the low bits of 1.5 2^23 + n): the conversion unit has a quarter of the rate.
constexpr float kRound = 12582912.f;
__device__ __forceinline__ void codes_of_row(const float (&r)[4], float sh, float zh, float inv, float maxq, float (&q)[4])
{
    float worst = 1.f;                               // least distance from a boundary, less the bound on the error
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float t = r[c] * inv, v = t + zh, w = fminf(fmaxf(v, -1.f), maxq + 1.f), n = (w + kRound) - kRound;
        worst = fminf(worst, (0.5f - fabsf(w - n)) - (fabsf(t) + fabsf(v)) * 6e-7f);
        q[c] = fminf(fmaxf(n, 0.f), maxq);
    }
    if (worst <= 0.f) {
#pragma unroll
        for (int c = 0; c < 4; ++c) q[c] = fminf(fmaxf(rintf(__fadd_rn(__fdiv_rn(r[c], sh), zh)), 0.f), maxq);
    }
}

// Eight consecutive values of T as floats.
__device__ __forceinline__ void widen8(const uint4 (&v)[1], float (&f)[8], const __half *)
{
    const __half2 *h = reinterpret_cast<const __half2 *>(v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 p = __half22float2(h[i]);
        f[2 * i] = p.x;
        f[2 * i + 1] = p.y;
    }
}
__device__ __forceinline__ void widen8(const uint4 (&v)[1], float (&f)[8], const __nv_bfloat16 *)
{
    const uint32_t w[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
}
__device__ __forceinline__ void widen8(const uint4 (&v)[2], float (&f)[8], const float *)
{
    memcpy(f, v, 32);
}

// vec: rows of B start on 16-byte boundaries (those of A always do)
template <typename T, bool kDelta>
__global__ void __launch_bounds__(kQThreads, 2)
quantise_tile_kernel(const float *__restrict__ W, const T *__restrict__ A, const T *__restrict__ B, uint8_t *__restrict__ codes,
                     __half *__restrict__ scales, __half *__restrict__ zeros, float *__restrict__ WF, float *__restrict__ Delta, int N, int K,
                     int bits, int rank, int vec)
{
    extern __shared__ __align__(16) uint8_t q_smem[];
    float4 *s_w = reinterpret_cast<float4 *>(q_smem);                         // [row of the warp][thread]
    float(*s_a)[kQT] = reinterpret_cast<float(*)[kQT]>(q_smem + kQSmemW);
    float(*s_b)[kQT] = reinterpret_cast<float(*)[kQT]>(q_smem + kQSmemW + kQSmemA);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = K / kQT, g = blockIdx.y, row0 = blockIdx.x * kQT;
    const size_t at0 = (size_t)g * kQT + 4 * lane;
    const int n0 = row0 + warp * 16;
#pragma unroll
    for (int i = 0; i < 16; ++i) ptx::cp_async16(ptx::smem_u32(s_w + i * kQThreads + tid), W + (size_t)min(n0 + i, N - 1) * K + at0);
    // chunks of eight values of A (16 per rank index) and of B (4 per row): two of each per thread
    constexpr int NV = (int)sizeof(T) / 2, kChunks = kQJ * 16;
    static_assert(kChunks == 2 * kQThreads && kQT * kQJ == 8 * kChunks, "two chunks of A and of B per thread");
    uint4 pa[2][NV], pb[2][NV];
    auto fetch = [&](int j0) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int e = tid + k * kQThreads;
            const int ja = j0 + (e >> 4), rb = row0 + (e & 127), jb = j0 + 8 * (e >> 7);
#pragma unroll
            for (int v = 0; v < NV; ++v) pa[k][v] = pb[k][v] = make_uint4(0u, 0u, 0u, 0u);
            if (ja < rank) {
                const uint4 *src = reinterpret_cast<const uint4 *>(A + (size_t)ja * K + (size_t)g * kQT + 8 * (e & 15));
#pragma unroll
                for (int v = 0; v < NV; ++v) pa[k][v] = __ldg(src + v);
            }
            if (rb < N && jb < rank) {
                const T *src = B + (size_t)rb * rank + jb;
                if (vec) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) pb[k][v] = __ldg(reinterpret_cast<const uint4 *>(src) + v);
                } else {
                    T *dst = reinterpret_cast<T *>(pb[k]);
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (jb + c < rank) dst[c] = src[c];
                }
            }
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int e = tid + k * kQThreads;
            float f[8];
            widen8(pa[k], f, static_cast<const T *>(nullptr));
            float4 *dst = reinterpret_cast<float4 *>(&s_a[e >> 4][8 * (e & 15)]);
            dst[0] = make_float4(f[0], f[1], f[2], f[3]);
            dst[1] = make_float4(f[4], f[5], f[6], f[7]);
            widen8(pb[k], f, static_cast<const T *>(nullptr));
#pragma unroll
            for (int c = 0; c < 8; ++c) s_b[8 * (e >> 7) + c][e & 127] = f[c];
        }
    };
    unsigned long long acc[8][4];                    // rows 2i and 2i + 1 (low and high word), k 4 lane + c
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0ull;
    if (rank > 0) fetch(0);
    for (int j0 = 0; j0 < rank; j0 += kQJ) {
        const int jn = min(kQJ, rank - j0);
        if (j0) __syncthreads();
        store();
        __syncthreads();
        if (j0 + kQJ < rank) fetch(j0 + kQJ);
#pragma unroll 4
        for (int j = 0; j < jn; ++j) {
            const float4 av = *reinterpret_cast<const float4 *>(&s_a[j][4 * lane]);
            const unsigned long long a[4] = {twice(av.x), twice(av.y), twice(av.z), twice(av.w)};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const Pair2 b = *reinterpret_cast<const Pair2 *>(&s_b[j][warp * 16 + 4 * q]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    fma2(acc[2 * q][c], b.x, a[c]);
                    fma2(acc[2 * q + 1][c], b.y, a[c]);
                }
            }
        }
    }
    ptx::cp_async_wait_all();                        // a thread reads only what it copied itself
    // r = W - Sigma
    float r[16][4], mn[16], mx[16];
    auto sigma = [&](int i, int c) { return __uint_as_float((unsigned)(acc[i >> 1][c] >> (32 * (i & 1)))); };
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float4 w = s_w[i * kQThreads + tid];
        r[i][0] = __fsub_rn(w.x, sigma(i, 0));
        r[i][1] = __fsub_rn(w.y, sigma(i, 1));
        r[i][2] = __fsub_rn(w.z, sigma(i, 2));
        r[i][3] = __fsub_rn(w.w, sigma(i, 3));
        mn[i] = fminf(fminf(r[i][0], r[i][1]), fminf(r[i][2], r[i][3]));
        mx[i] = fmaxf(fmaxf(r[i][0], r[i][1]), fmaxf(r[i][2], r[i][3]));
    }
#pragma unroll
    for (int step = 0; step < 4; ++step) {                     // 16 -> 8 -> 4 -> 2 -> 1 rows per lane, lane bits 4 .. 1
        const int o = 16 >> step, keep = 8 >> step;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < keep; ++i) {
            const float sn = up ? mn[i] : mn[i + keep], sx = up ? mx[i] : mx[i + keep];
            const float kn = up ? mn[i + keep] : mn[i], kx = up ? mx[i + keep] : mx[i];
            mn[i] = fminf(kn, __shfl_xor_sync(0xffffffffu, sn, o));
            mx[i] = fmaxf(kx, __shfl_xor_sync(0xffffffffu, sx, o));
        }
    }
    mn[0] = fminf(mn[0], __shfl_xor_sync(0xffffffffu, mn[0], 1));
    mx[0] = fmaxf(mx[0], __shfl_xor_sync(0xffffffffu, mx[0], 1));
    float s_row, z_row, inv_row;                               // of row lane / 2
    {
        const int n = n0 + (lane >> 1);
        __half s_h, z_h;
        scale_and_zero(mn[0], mx[0], bits, s_h, z_h);
        if (scales && !(lane & 1) && n < N) {
            scales[(size_t)n * G + g] = s_h;
            zeros[(size_t)n * G + g] = z_h;
        }
        s_row = __half2float(s_h);
        z_row = __half2float(z_h);
        inv_row = __frcp_rn(s_row);
    }
    const float maxq = (float)((1 << bits) - 1);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float sh = __shfl_sync(0xffffffffu, s_row, 2 * i), zh = __shfl_sync(0xffffffffu, z_row, 2 * i);
        float q[4];
        codes_of_row(r[i], sh, zh, __shfl_sync(0xffffffffu, inv_row, 2 * i), maxq, q);
        if (n0 + i >= N) continue;
        const size_t at = (size_t)(n0 + i) * K + at0;
        if (codes) {
            uint32_t b[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c] = __float_as_uint(q[c] + kRound);                // the code is the low byte
            *reinterpret_cast<uint32_t *>(codes + at) = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
        }
        if constexpr (kDelta) {
            const float4 w = s_w[i * kQThreads + tid];
            const float wv[4] = {w.x, w.y, w.z, w.w};
            float wf[4], d[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                wf[c] = __fadd_rn(__fmul_rn(sh, __fsub_rn(q[c], zh)), sigma(i, c));
                d[c] = __fsub_rn(wv[c], wf[c]);
            }
            if (WF) *reinterpret_cast<float4 *>(WF + at) = make_float4(wf[0], wf[1], wf[2], wf[3]);
            if (Delta) *reinterpret_cast<float4 *>(Delta + at) = make_float4(d[0], d[1], d[2], d[3]);
        }
    }
}

}  // namespace

// ab_kind: 0 = fp16, 1 = bf16, 2 = fp32 sub-branch matrices
cudaError_t launch_quantize_feedback(const float *W, const void *A, const void *B, uint8_t *codes, __half *scales,
                                     __half *zeros, float *WF, float *Delta, int N, int K, int group, int bits, int rank,
                                     int ab_kind, cudaStream_t s)
{
    auto go = [&](auto tag) {
        using T = decltype(tag);
        const T *a = static_cast<const T *>(A), *b = static_cast<const T *>(B);
        // 16-byte accesses of W and the fp32 outputs, 4-byte ones of the codes: K is a multiple of 128 here
        auto aligned = [](const void *q, unsigned n) { return (reinterpret_cast<uintptr_t>(q) & (n - 1)) == 0; };
        if (group == kQT && aligned(W, 16) && aligned(A, 16) && aligned(WF, 16) && aligned(Delta, 16) && aligned(codes, 4)) {
            const dim3 grid((unsigned)((N + kQT - 1) / kQT), (unsigned)(K / kQT));
            const int vec = aligned(B, 16) && ((size_t)rank * sizeof(T)) % 16 == 0 && rank % 8 == 0;
            auto kern = (WF || Delta) ? quantise_tile_kernel<T, true> : quantise_tile_kernel<T, false>;
            if (const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQSmem); e != cudaSuccess) return e;
            kern<<<grid, kQThreads, kQSmem, s>>>(W, a, b, codes, scales, zeros, WF, Delta, N, K, bits, rank, vec);
            return cudaGetLastError();
        }
        const dim3 grid((unsigned)N, (unsigned)(K / group));
        const unsigned block = (unsigned)((group + 31) / 32 * 32);
        quantize_feedback_kernel<T><<<grid, block, 0, s>>>(W, a, b, codes, scales, zeros, WF, Delta, N, K, group, bits, rank);
        return cudaGetLastError();
    };
    return ab_kind == 2 ? go(float{}) : ab_kind == 1 ? go(__nv_bfloat16{}) : go(__half{});
}

}  // namespace fbq

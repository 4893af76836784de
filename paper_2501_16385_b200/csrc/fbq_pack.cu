// Packing, unpacking and dense dequantisation kernels (offline / test aids of
// the weight-only quantised storage; Section 1 of the paper keeps weights in
// INT3/INT4).  One thread packs a run of 32 codes, or produces one code (unpack,
// dequant); all accesses are coalesced along K.
#include "fbq_common.cuh"

namespace fbq {
namespace {

// The packers move 8 (INT4) or 8/3 (INT3) times their output's bits and are bound by HBM: a thread takes a whole run of
// 32 codes with two 16-byte loads (a thread per packed word read them byte by byte: 11008 x 4096 INT3 took 22 us, now 8).
// Runs lie end to end whatever the row, since K is a multiple of 32; INT4 rows of other lengths end in single words.

// INT4: word w of a row takes codes 8w .. 8w+7, code e at bits 4e..4e+3.
__device__ __forceinline__ uint32_t pack8(uint32_t lo, uint32_t hi)
{
    lo &= 0x0F0F0F0Fu;
    hi &= 0x0F0F0F0Fu;
    lo |= lo >> 4;                                       // codes 0, 1 in byte 0; 2, 3 in byte 2
    hi |= hi >> 4;
    return __byte_perm(lo, hi, 0x6420);
}

__global__ void pack4_kernel(const uint8_t *__restrict__ codes, uint32_t *__restrict__ qw, size_t n_words)
{
    const size_t w = 4 * (blockIdx.x * (size_t)blockDim.x + threadIdx.x);
    if (w + 4 <= n_words) {
        const uint4 a = *reinterpret_cast<const uint4 *>(codes + 8 * w), b = *reinterpret_cast<const uint4 *>(codes + 8 * w + 16);
        *reinterpret_cast<uint4 *>(qw + w) = make_uint4(pack8(a.x, a.y), pack8(a.z, a.w), pack8(b.x, b.y), pack8(b.z, b.w));
        return;
    }
    for (size_t i = w; i < n_words; ++i) {
        const uint2 c = *reinterpret_cast<const uint2 *>(codes + 8 * i);
        qw[i] = pack8(c.x, c.y);
    }
}

// INT3: the three words of a 32-code run; word i:
//   fields f=0..4 at bits 3f: c[10i+f]; at bits 16+3f: c[10i+5+f];
//   bit 15: bit i of c[30]; bit 31: bit i of c[31].
__global__ void pack3_kernel(const uint8_t *__restrict__ codes, uint32_t *__restrict__ qw, size_t n_runs)
{
    const size_t run = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (run >= n_runs) return;
    const uint4 a = *reinterpret_cast<const uint4 *>(codes + 32 * run), b = *reinterpret_cast<const uint4 *>(codes + 32 * run + 16);
    const uint32_t c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    auto code = [&](int k) { return (c[k >> 2] >> (8 * (k & 3))) & 7u; };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        uint32_t w = ((code(30) >> i) & 1u) << 15 | ((code(31) >> i) & 1u) << 31;
#pragma unroll
        for (int f = 0; f < 5; ++f) w |= code(10 * i + f) << (3 * f) | code(10 * i + 5 + f) << (16 + 3 * f);
        qw[3 * run + i] = w;
    }
}

__device__ __forceinline__ uint32_t fetch_code(const uint32_t *__restrict__ qw, size_t row_words_base,
                                               int k, int bits)
{
    if (bits == 4) {
        const uint32_t w = qw[row_words_base + (k >> 3)];
        return (w >> ((k & 7) * 4)) & 0xFu;
    }
    const uint32_t *r = qw + row_words_base + (size_t)(k >> 5) * 3;
    const int c = k & 31;
    if (c >= 30) {
        const int sh = (c == 30) ? 15 : 31;
        return ((r[0] >> sh) & 1u) | (((r[1] >> sh) & 1u) << 1) | (((r[2] >> sh) & 1u) << 2);
    }
    const int i = c / 10, f = c - 10 * i;
    const int sh = (f < 5) ? 3 * f : 3 * f + 1;          // 16 + 3(f-5) = 3f + 1
    return (r[i] >> sh) & 7u;
}

__global__ void unpack_kernel(const uint32_t *__restrict__ qw, uint8_t *__restrict__ codes, int N, int K,
                              int bits)
{
    const size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (idx >= (size_t)N * K) return;
    const int n = (int)(idx / K), k = (int)(idx - (size_t)n * K);
    const size_t row_words = (bits == 4) ? (size_t)(K / 8) : (size_t)(K / 32) * 3;
    codes[idx] = (uint8_t)fetch_code(qw, n * row_words, k, bits);
}

__global__ void dequant_kernel(const uint32_t *__restrict__ qw, const __half *__restrict__ sc,
                               const __half *__restrict__ ze, float *__restrict__ W, int N, int K, int group,
                               int bits)
{
    const size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (idx >= (size_t)N * K) return;
    const int n = (int)(idx / K), k = (int)(idx - (size_t)n * K);
    const size_t row_words = (bits == 4) ? (size_t)(K / 8) : (size_t)(K / 32) * 3;
    const int G = K / group;
    const float s = __half2float(sc[(size_t)n * G + k / group]);
    const float z = __half2float(ze[(size_t)n * G + k / group]);
    const float q = (float)fetch_code(qw, n * row_words, k, bits);
    W[idx] = __fmul_rn(s, __fsub_rn(q, z));   // exact: 11-bit significand times a 5-bit integer
}

}  // namespace

cudaError_t launch_pack(const uint8_t *codes, uint32_t *qw, int N, int K, int bits, cudaStream_t s)
{
    const size_t n_words = (size_t)N * K / 8, n_runs = (size_t)N * K / 32;
    const int threads = 256;
    auto blocks = [&](size_t n) { return (unsigned)((n + threads - 1) / threads); };
    if (bits == 4)
        pack4_kernel<<<blocks((n_words + 3) / 4), threads, 0, s>>>(codes, qw, n_words);
    else
        pack3_kernel<<<blocks(n_runs), threads, 0, s>>>(codes, qw, n_runs);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const uint32_t *qw, uint8_t *codes, int N, int K, int bits, cudaStream_t s)
{
    const size_t total = (size_t)N * K;
    const int threads = 256;
    unpack_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, s>>>(qw, codes, N, K, bits);
    return cudaGetLastError();
}

cudaError_t launch_dequant(const uint32_t *qw, const __half *sc, const __half *ze, float *W, int N, int K,
                           int group, int bits, cudaStream_t s)
{
    const size_t total = (size_t)N * K;
    const int threads = 256;
    dequant_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, s>>>(qw, sc, ze, W, N, K, group,
                                                                                  bits);
    return cudaGetLastError();
}

}  // namespace fbq

// One iteration of layer-wise reconstruction (Algorithm 1 lines 5-9, Section 4.2 of the paper):
//
//   Delta_F = W - Q(W - B A) - B A                      (feedback quantiser of Section 4.1, detached)
//   L       = tr(Delta_F H Delta_F^T),  H = X^T X        (= ||W X^T - W_F X^T||_F^2)
//   G       = dL/dSigma = -2 Delta_F H
//   dL/dB   = G A^T,   dL/dA = B^T G                     (Sigma = B A)
//   A <- A - lr dL/dA,  B <- B - lr dL/dB                (both gradients from the old A, B)
//
// All matrices are fp32, and so are the products: each fp32 operand is cut into three bf16 terms (8 + 8 + 8 significant
// bits, exact), and the tensor cores multiply and add the six pairs of terms that reach fp32's last bit (the three left
// out are below 2^-26 of a product).  The tensor cores accumulate 64 terms of the leading pair at a time, which are then
// added to fp32 registers (rounded to nearest: they cut their own sums off, 4e-7 of a Gram matrix over 256 terms); the other
// five pairs, 2^-8 and smaller, have an accumulator of their own.  Against float64 the results are closer than those of the
// fp32 multiply-add loop this replaces (4096 x 4096, 4096 terms: 1.6e-7 against 9.9e-7, the steps 2e-7 against 1.6e-6).
//
// The order of the products is chosen for the work: neither gradient needs G (2 N K^2 operations) itself,
//   dL/dB = -2 Delta_F (H A^T),   dL/dA = -2 (B^T Delta_F) H          (four products of 2 N K r or 2 K^2 r)
// and the loss is the dot product of H with Delta_F^T Delta_F, which is symmetric: one triangle of it is enough.  H = X^T X is
// symmetric too (the Gram matrix here to the last bit), so that its rows serve as its columns and one triangle of it does for
// the loss; whether the caller's H is gets looked up while it is split, and where it is not its columns are split as well.
// 4096 x 4096, rank 128: the Gram matrix of 4096 tokens 5733 -> 320 us, the step 8099 -> 700 us.
#include <algorithm>

#include "fbq_common.cuh"
#include "fbq_maps.h"
#include "fbq_umma.cuh"

namespace fbq {
namespace {
using namespace ptx;

// ------------------------------------------------------------------ the product kernel
// C[m][n] = sum_k P[m][k] Q[n][k] over split operands [3 terms][rows][k].  Pairs of CTAs, persistent: 256 rows of P (128 per
// CTA) x `nt` rows of Q, one stage of 64 k holds all six terms (96 KB per CTA, two stages); 24 MMAs per stage take 3072
// cycles at nt = 256, so the loads (32 bytes per cycle) and the draining of the leading accumulator hide behind them: the
// tensor cores bound it.  Warps: 0 copies, 1 MMAs, 2 owns the tensor memory, 4-19 accumulate and write.
constexpr int kBK = 64, kRows = 256, kStages = 2, kTerms = 3;
constexpr uint32_t kTermBytes = 128u * kBK * 2u, kStageBytes = 2u * kTerms * kTermBytes;
constexpr int kEpi = 4, kEpiWarps = 16, kThreads = (kEpi + kEpiWarps) * 32;
constexpr uint32_t kBarOff = kStages * kStageBytes;
constexpr size_t kSmem = kBarOff + (2 * kStages + 4) * 8u + 64u;
constexpr int kPromote = 1;                      // stages between additions of the leading accumulator to registers
constexpr uint32_t kSmallCol = 256;              // tensor-memory column of the other accumulator

enum Mode { kSymmetric, kDot, kPartial };        // write both triangles; dot product with H; one slice per split of k
struct ProductParams {
    float *C;                 // kSymmetric: [n][n]; kPartial: [split][M][N]
    int add;                  // kSymmetric: add to C
    const float *H;           // kDot
    const int *skew;          // kDot: not zero if H is not symmetric
    double *dots;             // kDot: [work item][CTA][warp]
    int *status;
    int M, N, K;
    int nt;                   // rows of Q per tile (a multiple of 32, at most 256)
    int tiles_m, tiles_n, splits;
};

// work item q -> tile and range of stages
__device__ __forceinline__ void locate(const ProductParams &p, int mode, int q, int &tm, int &tn, int &split, int &kb0, int &kb1)
{
    const int kb = (p.K + kBK - 1) / kBK;
    if (mode == kPartial) {
        split = q % p.splits;
        tn = q / p.splits % p.tiles_n;
        tm = q / p.splits / p.tiles_n;
    } else {                                     // triangle: tm <= tn
        split = 0;
        tn = (int)((sqrtf(8.f * (float)q + 1.f) - 1.f) * 0.5f);
        while (tn * (tn + 1) / 2 > q) --tn;
        while ((tn + 1) * (tn + 2) / 2 <= q) ++tn;
        tm = q - tn * (tn + 1) / 2;
    }
    kb0 = (int)((long long)split * kb / p.splits);
    kb1 = (int)((long long)(split + 1) * kb / p.splits);
}

__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t cluster_bar)
{
    asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
                 "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(cluster_bar)
                 : "memory");
}

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
product_kernel(const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap qmap, const ProductParams p, const int n_work)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const uint32_t full0 = sbase + kBarOff, empty0 = full0 + 8u * kStages, hfull = empty0 + 8u * kStages, hfree = hfull + 8u, sfull = hfree + 8u,
                   sfree = sfull + 8u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kBarOff + (2 * kStages + 4) * 8u);
    volatile int *quit = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t cr = cluster_ctarank();
    const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
    pdl_launch_dependents();
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full0 + 8u * i, 1);
            mbar_init(empty0 + 8u * i, 1);
        }
        mbar_init(hfull, 1);
        mbar_init(hfree, 2 * kEpiWarps);
        mbar_init(sfull, 1);
        mbar_init(sfree, 2 * kEpiWarps);
        *quit = 0;
        fence_barrier_init();
    }
    if (warp == 2) umma::tmem_alloc<2>(smem_u32(tmem_slot), 512);
    umma::fence_before();
    cluster_arrive();
    cluster_wait();
    umma::fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    pdl_wait();                                                  // all of the above overlaps the preceding kernel

    if (warp == 0) {
        if (lane == 0) {
            const uint32_t lfull0 = mapa_shared(full0, 0);
            const uint32_t q_bytes = (uint32_t)(p.nt / 2) * (kBK * 2u), bytes = 2u * kTerms * (kTermBytes + q_bytes);
            uint32_t i = 0;
            for (int q = pair; q < n_work && ok; q += n_pairs) {
                int tm, tn, split, kb0, kb1;
                locate(p, MODE, q, tm, tn, split, kb0, kb1);
                const int prow = tm * kRows + 128 * (int)cr, qrow = tn * p.nt + p.nt / 2 * (int)cr;
                for (int kb = kb0; kb < kb1; ++kb, ++i) {
                    const uint32_t s = i % kStages;
                    if (i >= (uint32_t)kStages && !umma::wait_cluster(empty0 + 8u * s, (i / kStages - 1u) & 1u, quit)) { ok = false; break; }
                    if (cr == 0) mbar_expect_tx(full0 + 8u * s, bytes);
                    const uint32_t at = sbase + s * kStageBytes;
#pragma unroll
                    for (int t = 0; t < kTerms; ++t) {
                        tma_load_3d_pair(at + t * kTermBytes, &pmap, kb * kBK, prow, t, lfull0 + 8u * s);
                        tma_load_3d_pair(at + (kTerms + t) * kTermBytes, &qmap, kb * kBK, qrow, t, lfull0 + 8u * s);
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (cr == 0 && lane == 0) {
            const uint32_t idesc = umma::idesc_f16(1, kRows, (uint32_t)p.nt);
            const uint64_t desc0 = umma::desc_k128(sbase);
            uint32_t i = 0, it = 0, drained = 0;
            for (int q = pair; q < n_work && ok; q += n_pairs, ++it) {
                int tm, tn, split, kb0, kb1;
                locate(p, MODE, q, tm, tn, split, kb0, kb1);
                for (int kb = kb0; kb < kb1; ++kb, ++i) {
                    const uint32_t s = i % kStages;
                    const int rel = kb - kb0;
                    if (!umma::wait_cluster(full0 + 8u * s, (i / kStages) & 1u, quit)) { ok = false; break; }
                    if (rel % kPromote == 0 && drained > 0 && !umma::wait_cluster(hfree, (drained - 1u) & 1u, quit)) { ok = false; break; }
                    umma::fence_after();
                    const uint64_t pd = desc0 + s * (kStageBytes >> 4), qd = pd + kTerms * (kTermBytes >> 4);
                    auto mul = [&](uint32_t d, int a, int b, bool fresh) {
#pragma unroll
                        for (int j = 0; j < kBK / 16; ++j)
                            umma::mma_pair(d, pd + a * (kTermBytes >> 4) + 2 * j, qd + b * (kTermBytes >> 4) + 2 * j, idesc, (fresh && j == 0) ? 0u : 1u);
                    };
                    mul(tmem, 0, 0, rel % kPromote == 0);
                    if (rel % kPromote == kPromote - 1 || kb == kb1 - 1) {
                        umma::commit_pair(hfull);
                        ++drained;
                    }
                    if (rel == 0 && it > 0 && !umma::wait_cluster(sfree, (it - 1u) & 1u, quit)) { ok = false; break; }
                    umma::fence_after();
                    mul(tmem + kSmallCol, 0, 2, rel == 0);
                    mul(tmem + kSmallCol, 2, 0, false);
                    mul(tmem + kSmallCol, 1, 1, false);
                    mul(tmem + kSmallCol, 0, 1, false);
                    mul(tmem + kSmallCol, 1, 0, false);
                    umma::commit_pair(empty0 + 8u * s);
                }
                if (ok) umma::commit_pair(sfull);
            }
        }
    } else if (warp >= kEpi) {
        const int wq = warp & 3, cw = p.nt / 4, c0 = ((warp - kEpi) >> 2) * cw;       // this warp's columns of a tile
        const uint32_t src = tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)c0, lhfree = mapa_shared(hfree, 0), lsfree = mapa_shared(sfree, 0);
        uint32_t it = 0, drained = 0;
        for (int q = pair; q < n_work && ok; q += n_pairs, ++it) {
            int tm, tn, split, kb0, kb1;
            locate(p, MODE, q, tm, tn, split, kb0, kb1);
            float acc[64];
#pragma unroll
            for (int j = 0; j < 64; ++j) acc[j] = 0.f;
            auto add = [&](uint32_t col, uint32_t bar) {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    if (16 * h < cw) {
                        uint32_t v[16];
                        umma::ld16(src + col + 16u * h, v);
                        umma::wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; ++j) acc[16 * h + j] += __uint_as_float(v[j]);
                    }
                }
                umma::fence_before();
                __syncwarp();
                if (lane == 0) umma::arrive_cluster(bar);
            };
            for (int kb = kb0; kb < kb1; kb += kPromote, ++drained) {
                if (!umma::wait_cluster(hfull, drained & 1u, quit)) { ok = false; break; }
                umma::fence_after();
                add(0, lhfree);
            }
            if (!ok || !umma::wait_cluster(sfull, it & 1u, quit)) { ok = false; break; }
            umma::fence_after();
            add(kSmallCol, lsfree);
            const int m = tm * kRows + 128 * (int)cr + 32 * wq + lane, n0 = tn * p.nt + c0;
            if constexpr (MODE == kDot) {
                // the tile times H's at (n, m), where the lanes read side by side; off the diagonal the same again for (m, n), or,
                // where H is not symmetric, the tile times that, a lane a row: whole sectors at a time where they are aligned
                const bool twice = tm != tn && *p.skew == 0, both = tm != tn && !twice;
                double dot = 0.0;
                const bool wide = (p.N & 7) == 0 && (reinterpret_cast<uintptr_t>(p.H) & 31u) == 0u;
#pragma unroll
                for (int j = 0; j < 64; j += 8) {
                    float part = 0.f, other = 0.f, h[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (j + e < cw && n0 + j + e < p.N && m < p.M) part = fmaf(acc[j + e], p.H[(size_t)(n0 + j + e) * p.M + m], part);
                    if (both && j < cw && n0 + j < p.N && m < p.M) {
                        const float *row = p.H + (size_t)m * p.N + n0 + j;
                        if (wide) {
                            *reinterpret_cast<float4 *>(h) = __ldg(reinterpret_cast<const float4 *>(row));
                            *reinterpret_cast<float4 *>(h + 4) = __ldg(reinterpret_cast<const float4 *>(row) + 1);
                        } else {
#pragma unroll
                            for (int e = 0; e < 8; ++e) h[e] = n0 + j + e < p.N ? row[e] : 0.f;
                        }
#pragma unroll
                        for (int e = 0; e < 8; ++e) other = fmaf(acc[j + e], h[e], other);
                    }
                    dot += (double)part;
                    dot += (double)other;
                }
                for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                if (lane == 0) p.dots[((size_t)q * 2 + cr) * kEpiWarps + (warp - kEpi)] = twice ? 2.0 * dot : dot;
            } else {
                const size_t pitch = (size_t)p.N;
                float *row = p.C + (MODE == kPartial ? (size_t)split * p.M * pitch : 0) + (size_t)m * pitch + n0;
                // (a tile on the diagonal holds both triangles, which differ in the last bits; the upper one is written twice)
                const bool on_diagonal = MODE == kSymmetric && tm == tn;
                if (MODE == kSymmetric && p.add && m < p.M) {
#pragma unroll
                    for (int j = 0; j < 64; ++j)
                        if (j < cw && n0 + j < p.N && (!on_diagonal || n0 + j >= m)) acc[j] += row[j];
                }
                if (m < p.M) {
#pragma unroll
                    for (int j = 0; j < 64; j += 4) {
                        if (on_diagonal && n0 + j < m) {
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (j < cw && n0 + j + e >= m && n0 + j + e < p.N) row[j + e] = acc[j + e];
                            continue;
                        }
                        if (j >= cw || n0 + j >= p.N) break;
                        if (n0 + j + 3 < p.N && (pitch & 3u) == 0u && (reinterpret_cast<uintptr_t>(p.C) & 15u) == 0u) {
                            *reinterpret_cast<float4 *>(row + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
                        } else {
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (n0 + j + e < p.N) row[j + e] = acc[j + e];
                        }
                    }
                    if (MODE == kSymmetric) {
#pragma unroll
                        for (int j = 0; j < 64; ++j)
                            if (j < cw && n0 + j < p.N && n0 + j > m) p.C[(size_t)(n0 + j) * pitch + m] = acc[j];
                    }
                }
            }
        }
    }
    if (!ok) {
        *quit = 1;
        if (p.status) atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
        for (int i = 0; i < 64; ++i) __nanosleep(1000);          // copies in flight land before the CTA leaves
    }
    umma::fence_before();
    __syncthreads();
    cluster_arrive();
    cluster_wait();
    if (warp == 2) {
        umma::fence_after();
        umma::tmem_free<2>(tmem, 512);
    }
}

// ------------------------------------------------------------------ operands
// x = h + m + l, three bf16 terms (round to nearest, so each is at most 2^-9 of the one before; exact for 24 bits).
__device__ __forceinline__ void terms(float x, unsigned short (&t)[kTerms])
{
#pragma unroll
    for (int i = 0; i < kTerms; ++i) {
        const __nv_bfloat16 b = __float2bfloat16_rn(x);
        t[i] = __bfloat16_as_ushort(b);
        x -= __bfloat162float(b);
    }
}
__device__ __forceinline__ void store_terms(unsigned short *dst, size_t plane, const float (&v)[4], int count)
{
    unsigned short t[4][kTerms];
#pragma unroll
    for (int e = 0; e < 4; ++e) terms(v[e], t[e]);
#pragma unroll
    for (int i = 0; i < kTerms; ++i) {
        if (count >= 4) {
            *reinterpret_cast<ushort4 *>(dst + i * plane) = make_ushort4(t[0][i], t[1][i], t[2][i], t[3][i]);
        } else {
            for (int e = 0; e < count; ++e) dst[i * plane + e] = t[e][i];
        }
    }
}
// The matrix [R][C] (rows `ld` apart) as terms, rows as they are (`rows`: [3][R][pitch_r]) and / or transposed (`cols`: [3][C][pitch_c]).  Bound
// by HBM: 4 bytes read, 6 written per copy and element; 64 x 64 tiles through shared memory, 8-byte stores.
__device__ __forceinline__ void split_tile(const float *__restrict__ src, size_t ld, int R, int C, unsigned short *rows, size_t pitch_r,
                                           unsigned short *cols, size_t pitch_c, int tile_r, int tile_c)
{
    __shared__ float tile[64][65];
    const int r0 = tile_r * 64, c0 = tile_c * 64, tid = threadIdx.x;
    if (r0 >= R || c0 >= C) return;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int e = tid + 256 * i, r = e >> 6, c = e & 63;
        tile[r][c] = (r0 + r < R && c0 + c < C) ? src[(r0 + r) * ld + c0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = tid + 256 * i, a = e >> 4, b = (e & 15) * 4;
        if (rows && r0 + a < R && c0 + b < C) {
            const float v[4] = {tile[a][b], tile[a][b + 1], tile[a][b + 2], tile[a][b + 3]};
            store_terms(rows + (size_t)(r0 + a) * pitch_r + c0 + b, (size_t)R * pitch_r, v, C - (c0 + b));
        }
        if (cols && c0 + a < C && r0 + b < R) {
            const float v[4] = {tile[b][a], tile[b + 1][a], tile[b + 2][a], tile[b + 3][a]};
            store_terms(cols + (size_t)(c0 + a) * pitch_c + r0 + b, (size_t)C * pitch_c, v, R - (r0 + b));
        }
    }
}

__global__ void __launch_bounds__(256) split_kernel(const float *__restrict__ src, size_t ld, int R, int C, unsigned short *rows, size_t pitch_r,
                                                    unsigned short *cols, size_t pitch_c)
{
    split_tile(src, ld, R, C, rows, pitch_r, cols, pitch_c, blockIdx.y, blockIdx.x);
}
// A transposed split that is done if `wanted` says so (most launches only look).
struct SplitIf {
    const float *src;
    size_t ld;
    int R, C;
    unsigned short *cols;
    size_t pitch;
    const int *wanted;
};
__device__ __forceinline__ void split_if(const SplitIf &w, int block, int blocks)
{
    if (*w.wanted == 0) return;
    const int across = (w.C + 63) / 64, tiles = across * ((w.R + 63) / 64);
    for (int i = block; i < tiles; i += blocks) {
        split_tile(w.src, w.ld, w.R, w.C, nullptr, 0, w.cols, w.pitch, i / across, i % across);
        __syncthreads();
    }
}
// The sub-branch's A [r][K] as it is and B [N][r] transposed, and a flag cleared: one launch, since small layers are bound by
// the number of them.
__global__ void __launch_bounds__(256) split_branch_kernel(const float *__restrict__ A, int K, unsigned short *a_rows, size_t a_pitch,
                                                           const float *__restrict__ B, int N, unsigned short *b_cols, size_t b_pitch, int r, int *flag)
{
    const int ka = (K + 63) / 64, ra = (r + 63) / 64, i = blockIdx.x - ka * ra;
    if (i < 0) split_tile(A, K, r, K, a_rows, a_pitch, nullptr, 0, blockIdx.x / ka, blockIdx.x % ka);
    else split_tile(B, r, N, r, nullptr, 0, b_cols, b_pitch, i / ra, i % ra);
    if (i == 0 && threadIdx.x == 0) *flag = 0;
}

// The square matrix [K][K] as terms, rows as they are (not wanted: NULL); `skew` (cleared before) is raised if any two entries
// across the diagonal differ.  A block takes a tile and its mirror image (the blocks of the other triangle leave); a thread
// holds four quads of each and meets the mirrored values in shared memory.
__global__ void __launch_bounds__(256) split_square_kernel(const float *__restrict__ src, int K, unsigned short *rows, size_t pitch, int *skew)
{
    __shared__ float mirror[64][65];
    if (blockIdx.x < blockIdx.y) return;
    const int at[2] = {(int)blockIdx.y * 64, (int)blockIdx.x * 64}, tid = threadIdx.x;
    const bool wide = (K & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0u;
    float v[2][4][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = tid + 256 * i, r = at[h] + (e >> 4), c = at[1 - h] + (e & 15) * 4;
            if (wide && r < K && c < K) {
                *reinterpret_cast<float4 *>(v[h][i]) = __ldg(reinterpret_cast<const float4 *>(src + (size_t)r * K + c));
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) v[h][i][k] = (r < K && c + k < K) ? src[(size_t)r * K + c + k] : 0.f;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = tid + 256 * i;
#pragma unroll
        for (int k = 0; k < 4; ++k) mirror[e >> 4][(e & 15) * 4 + k] = v[1][i][k];
    }
    __syncthreads();
    bool differ = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = tid + 256 * i;
#pragma unroll
        for (int k = 0; k < 4; ++k) differ = differ || __float_as_uint(v[0][i][k]) != __float_as_uint(mirror[(e & 15) * 4 + k][e >> 4]);
    }
    if (__any_sync(0xffffffffu, differ) && (tid & 31) == 0) *skew = 1;
    if (!rows) return;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && blockIdx.x == blockIdx.y) break;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = tid + 256 * i, r = at[h] + (e >> 4), c = at[1 - h] + (e & 15) * 4;
            if (r < K && c < K) store_terms(rows + (size_t)r * pitch + c, (size_t)K * pitch, v[h][i], K - c);
        }
    }
}

// Sums the slices of a product [split][R][r] in order; transposed to terms [3][r][pitch], or added to `into` (rows `into_ld` apart) times alpha.
// Blocks of a second layer of the grid do `then`, which needs the product to have been read as well and is no launch of its own.
__global__ void __launch_bounds__(256) sum_transposed_kernel(const float *__restrict__ part, int splits, int R, int r, unsigned short *planes, size_t pitch,
                                                             float *into, size_t into_ld, float alpha, const SplitIf then)
{
    if (blockIdx.z) {
        split_if(then, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
        return;
    }
    __shared__ float tile[32][33];
    const int k0 = blockIdx.x * 32, j0 = blockIdx.y * 32, tid = threadIdx.x;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = (tid >> 5) + 8 * i, j = tid & 31;
        float v = 0.f;
        if (k0 + k < R && j0 + j < r)
            for (int s = 0; s < splits; ++s) v += part[((size_t)s * R + k0 + k) * r + j0 + j];
        tile[k][j] = v;
    }
    __syncthreads();
    const int j = tid >> 3, k = (tid & 7) * 4;
    if (j0 + j >= r || k0 + k >= R) return;
    const float v[4] = {tile[k][j], tile[k + 1][j], tile[k + 2][j], tile[k + 3][j]};
    if (planes) {
        store_terms(planes + (size_t)(j0 + j) * pitch + k0 + k, (size_t)r * pitch, v, R - (k0 + k));
    } else {
        for (int e = 0; e < 4 && k0 + k + e < R; ++e) {
            float *a = into + (j0 + j) * into_ld + k0 + k + e;
            *a = fmaf(alpha, v[e], *a);
        }
    }
}
__global__ void __launch_bounds__(256) sum_into_kernel(const float *__restrict__ part, int splits, size_t n, float *__restrict__ into, float alpha)
{
    const size_t i = blockIdx.x * (size_t)256 + threadIdx.x;
    if (i >= n) return;
    float v = 0.f;
    for (int s = 0; s < splits; ++s) v += part[s * n + i];
    into[i] = fmaf(alpha, v, into[i]);
}
// The loss: the work items' dot products added in a fixed order.
__global__ void __launch_bounds__(256) sum_dots_kernel(const double *__restrict__ dots, int n, float *out)
{
    __shared__ double sh[256];
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) v += dots[i];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = (float)sh[0];
}

// ------------------------------------------------------------------ host side
struct Operand {
    unsigned short *planes;   // [3][rows][pitch]
    int rows, k;
    size_t full_pitch = 0;    // of the operand that this is a range of k of (k_range); 0: all of it
    size_t pitch() const { return full_pitch ? full_pitch : ((size_t)k + 7) & ~(size_t)7; }
    size_t values() const { return (size_t)kTerms * rows * pitch(); }
    Operand k_range(int k0, int n) const { return Operand{planes + k0, rows, n, pitch()}; }      // k0: a multiple of 8
    Operand first(int n_rows, int n) const { return Operand{planes, n_rows, n}; }               // the same memory, smaller
};
cudaError_t operand_map(CUtensorMap *map, const Operand &o, int box_rows)
{
    MapSpec m{};
    m.base = o.planes;
    m.type = CU_TENSOR_MAP_DATA_TYPE_UINT16;
    m.ndim = 3;
    m.dims[0] = (cuuint64_t)o.k; m.dims[1] = (cuuint64_t)o.rows; m.dims[2] = kTerms;
    m.strides[0] = o.pitch() * 2; m.strides[1] = (cuuint64_t)o.rows * o.pitch() * 2;
    m.box[0] = kBK; m.box[1] = (cuuint32_t)box_rows; m.box[2] = 1;
    m.swizzle = CU_TENSOR_MAP_SWIZZLE_128B;
    return encode_map(map, m);
}

int pairs()
{
    static int n = 0;
    if (n == 0) {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 74;
        n = std::max(1, sms / 2);
    }
    return n;
}
// Slices of k for a product of few tiles: about one work item per pair, at least four stages each.
int k_splits(int M, int N, int K)
{
    const int tiles = ((M + kRows - 1) / kRows) * ((N + 255) / 256), kb = (K + kBK - 1) / kBK;
    return std::max(1, std::min(std::min(pairs() / tiles, kb / 4), 32));
}
int triangle_items(int n)
{
    const int t = (n + kRows - 1) / kRows;
    return t * (t + 1) / 2;
}

template <int MODE>
bool product(cudaStream_t s, const Operand &P, const Operand &Q, ProductParams p, bool pdl)
{
    p.M = P.rows; p.N = Q.rows; p.K = P.k;
    p.nt = MODE == kPartial ? std::min(256, (p.N + 31) / 32 * 32) : 256;
    p.tiles_m = (p.M + kRows - 1) / kRows;
    p.tiles_n = (p.N + p.nt - 1) / p.nt;
    p.splits = MODE == kPartial ? k_splits(p.M, p.N, p.K) : 1;
    const int n_work = MODE == kPartial ? p.tiles_m * p.tiles_n * p.splits : triangle_items(p.M);
    CUtensorMap pmap, qmap;
    if (operand_map(&pmap, P, 128) != cudaSuccess || operand_map(&qmap, Q, p.nt / 2) != cudaSuccess) return false;
    auto kern = product_kernel<MODE>;
    static bool attr_set = false;
    if (!attr_set) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem) != cudaSuccess) return false;
        attr_set = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(2 * std::min(pairs(), n_work)));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, pmap, qmap, p, n_work) == cudaSuccess;
}
bool split(cudaStream_t s, const float *src, size_t ld, int R, int C, const Operand *rows, const Operand *cols)
{
    const dim3 grid((unsigned)((C + 63) / 64), (unsigned)((R + 63) / 64));
    split_kernel<<<grid, 256, 0, s>>>(src, ld, R, C, rows ? rows->planes : nullptr, rows ? rows->pitch() : 0, cols ? cols->planes : nullptr, cols ? cols->pitch() : 0);
    return cudaGetLastError() == cudaSuccess;
}

bool split_square(cudaStream_t s, const float *src, int K, const Operand *rows, int *skew)
{
    const unsigned tiles = (unsigned)((K + 63) / 64);
    split_square_kernel<<<dim3(tiles, tiles), 256, 0, s>>>(src, K, rows ? rows->planes : nullptr, rows ? rows->pitch() : 0, skew);
    return cudaGetLastError() == cudaSuccess;
}

// Carves a call's scratch out of one block.
struct Carver {
    char *base;
    size_t used = 0;
    void *take(size_t bytes)
    {
        void *p = base ? base + used : nullptr;
        used += (bytes + 255) & ~(size_t)255;
        return p;
    }
    Operand operand(int rows, int k)
    {
        Operand o{nullptr, rows, k};
        o.planes = static_cast<unsigned short *>(take(o.values() * 2));
        return o;
    }
};
// Scratch is bounded: where the split operands of all of Delta_F, H or X would take more than `budget` bytes, they are split and
// multiplied a slab of rows at a time (kSlab rows at least).  What the rank needs comes on top.
constexpr int kSlab = kRows;
int slab_rows(int rows, size_t bytes_per_row, size_t budget)
{
    const size_t most = std::max((size_t)kSlab, budget / bytes_per_row / kSlab * kSlab), n = ((size_t)rows + most - 1) / most;
    return (int)std::min((size_t)rows, (((size_t)rows + n - 1) / n + kSlab - 1) / kSlab * kSlab);
}
struct StepScratch {
    int nd, nh;                             // rows of a slab of Delta_F and of H
    bool one_d;                             // Delta_F and its transpose one after the other in the same place
    Operand D, Dt, H, A, Bt, P, Q;          // slabs of Delta_F, its transpose and H; A, B^T, (H A^T)^T, (B^T Delta_F)
    float *part, *q_sum;                    // partial products; their sum over slabs of Delta_F where there are several
    double *dots;
    int *skew;
    size_t bytes;
    StepScratch(void *base, int N, int K, int r, size_t budget)
    {
        const size_t per_row = 2u * kTerms * (size_t)((K + 7) & ~7);        // bytes of one row's terms
        one_d = per_row * (2 * (size_t)N + K) > budget;
        nd = one_d ? slab_rows(N, per_row, budget / 2) : N;
        nh = one_d ? slab_rows(K, per_row, budget - std::min(budget / 2, per_row * nd)) : K;
        const int slabs = (N + nd - 1) / nd;
        Carver c{static_cast<char *>(base)};
        D = c.operand(nd, K);
        Dt = Operand{nullptr, K, nd};
        if (!one_d) Dt = c.operand(K, nd);
        else if (Dt.values() > D.values()) c.take((Dt.values() - D.values()) * 2);              // (rows of nd values are padded to 16 bytes)
        if (one_d) Dt.planes = D.planes;
        H = c.operand(nh, K);
        A = c.operand(r, K);
        Bt = c.operand(r, N);
        P = c.operand(r, K);
        Q = c.operand(r, K);
        // splits x rows of a product: a work item per pair and kRows rows each, or one split
        part = static_cast<float *>(c.take((size_t)std::max(std::max(K, N), pairs() * kRows) * r * sizeof(float)));
        q_sum = static_cast<float *>(c.take(slabs > 1 ? (size_t)K * r * sizeof(float) : 0));
        dots = static_cast<double *>(c.take((size_t)slabs * triangle_items(K) * 2 * kEpiWarps * sizeof(double)));
        skew = static_cast<int *>(c.take(sizeof(int)));
        bytes = c.used;
    }
};
}  // namespace

size_t reconstruct_workspace_floats(int N, int K, int rank)
{
    return 2 * (size_t)N * K + (size_t)rank * K + (size_t)N * rank + 256;
}

int gram_slab(int T, int K, size_t budget) { return slab_rows(T, 2u * kTerms * (size_t)K, budget); }
size_t gram_scratch_bytes(int T, int K, size_t budget)
{
    Carver c{nullptr};
    c.operand(K, gram_slab(T, K, budget));
    return c.used;
}
size_t reconstruct_scratch_bytes(int N, int K, int rank, size_t budget) { return StepScratch(nullptr, N, K, rank, budget).bytes; }

// H[K x K] = X^T X for X [T x K]; several slabs of X are added one after the other
int run_gram(const float *X, float *H, int T, int K, size_t budget, void *scratch, int *status, bool pdl, cudaStream_t s, int *launches)
{
    const int nt = gram_slab(T, K, budget);
    Carver c{static_cast<char *>(scratch)};
    const Operand all = c.operand(K, nt);
    ProductParams p{};
    p.C = H;
    p.status = status;
    for (int t0 = 0; t0 < T; t0 += nt) {
        const Operand Xt = all.first(K, std::min(nt, T - t0));
        p.add = t0 > 0;
        if (!split(s, X + (size_t)t0 * K, K, Xt.k, K, nullptr, &Xt) || !product<kSymmetric>(s, Xt, Xt, p, pdl)) return FBQ_ERR_CUDA;
        *launches += 2;
    }
    return FBQ_OK;
}

int run_reconstruct_step(const float *W, const float *H, float *A, float *B, float lr, float *loss, float *ws, int N, int K, int group, int bits,
                         int rank, size_t budget, void *scratch, int *status, bool pdl, cudaStream_t s, int *launches)
{
    const StepScratch t(scratch, N, K, rank, budget);
    const int slabs_d = (N + t.nd - 1) / t.nd, slabs_h = (K + t.nh - 1) / t.nh, items = triangle_items(K) * 2 * kEpiWarps;
    const size_t nq = (size_t)K * rank;
    ProductParams p{};
    p.status = status;
    p.C = t.part;
    p.skew = t.skew;
    bool ok = true;
    auto columns = [&](const float *part, int splits, int rows, unsigned short *planes, size_t pitch, float *into, float alpha, const SplitIf *then = nullptr) {
        const dim3 grid((unsigned)((rows + 31) / 32), (unsigned)((rank + 31) / 32), then ? 2u : 1u);
        sum_transposed_kernel<<<grid, 256, 0, s>>>(part, splits, rows, rank, planes, pitch, into, (size_t)K, alpha, then ? *then : SplitIf{});
        ++*launches;
    };
    auto add = [&](const float *part, int splits, size_t n, float *into, float alpha) {
        sum_into_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, splits, n, into, alpha);
        ++*launches;
    };
    auto times = [&](const Operand &P, const Operand &Q) {      // -> number of splits in t.part
        ok = ok && product<kPartial>(s, P, Q, p, pdl);
        ++*launches;
        return k_splits(P.rows, Q.rows, P.k);
    };
    // Delta_F with Q(W - B A) held fixed (nothing else of the quantiser's output is kept)
    float *Delta = ws;
    if (launch_quantize_feedback(W, A, B, nullptr, nullptr, nullptr, nullptr, Delta, N, K, group, bits, rank, 2, s) != cudaSuccess) return FBQ_ERR_CUDA;
    split_branch_kernel<<<(unsigned)(((rank + 63) / 64) * ((K + 63) / 64 + (N + 63) / 64)), 256, 0, s>>>(
        A, K, t.A.planes, t.A.pitch(), B, N, t.Bt.planes, t.Bt.pitch(), rank, t.skew);
    ok = split_square(s, H, K, slabs_h == 1 ? &t.H : nullptr, t.skew);
    *launches += 3;
    // slabs of Delta_F, transposed: the loss tr(Delta H Delta^T) = sum H o (Delta^T Delta), elementwise, and Delta^T B [K x rank]
    if (slabs_d > 1) ok = ok && cudaMemsetAsync(t.q_sum, 0, nq * sizeof(float), s) == cudaSuccess;
    for (int i = 0; i < slabs_d && ok; ++i) {
        const int n0 = i * t.nd, n = std::min(t.nd, N - n0);
        const Operand D = t.D.first(n, K), Dt = t.Dt.first(K, n);
        ok = split(s, Delta + (size_t)n0 * K, K, n, K, t.one_d ? nullptr : &D, &Dt);
        ++*launches;
        if (loss) {
            ProductParams d = p;
            d.H = H;
            d.dots = t.dots + (size_t)i * items;
            ok = ok && product<kDot>(s, Dt, Dt, d, pdl);
            ++*launches;
        }
        const int splits = times(Dt, t.Bt.k_range(n0, n));
        if (slabs_d > 1) add(t.part, splits, nq, t.q_sum, 1.f);
        else columns(t.part, splits, K, t.Q.planes, t.Q.pitch(), nullptr, 0.f);
    }
    if (slabs_d > 1) columns(t.q_sum, 1, K, t.Q.planes, t.Q.pitch(), nullptr, 0.f);
    if (loss) {
        sum_dots_kernel<<<1, 256, 0, s>>>(t.dots, slabs_d * items, loss);
        ++*launches;
    }
    // Slabs of H: H A^T [K x rank] from its rows; A <- A + 2 lr (B^T Delta) H from its columns, which take the rows' place unless
    // H is symmetric and they are the same (A and B enter as they were: their terms are made above).
    for (int i = 0; i < slabs_h && ok; ++i) {
        const int k0 = i * t.nh, n = std::min(t.nh, K - k0);
        const Operand Hs = t.H.first(n, K);
        if (slabs_h > 1) {
            ok = split(s, H + (size_t)k0 * K, K, n, K, &Hs, nullptr);
            ++*launches;
        }
        const SplitIf cols{H + k0, (size_t)K, K, n, Hs.planes, Hs.pitch(), t.skew};
        columns(t.part, times(Hs, t.A), n, t.P.planes + k0, t.P.pitch(), nullptr, 0.f, &cols);
        columns(t.part, times(Hs, t.Q), n, nullptr, 0, A + k0, 2.f * lr);
    }
    // slabs of Delta_F: B <- B + 2 lr Delta (H A^T)
    for (int i = 0; i < slabs_d && ok; ++i) {
        const int n0 = i * t.nd, n = std::min(t.nd, N - n0);
        const Operand D = t.D.first(n, K);
        if (t.one_d) {
            ok = split(s, Delta + (size_t)n0 * K, K, n, K, &D, nullptr);
            ++*launches;
        }
        add(t.part, times(D, t.P), (size_t)n * rank, B + (size_t)n0 * rank, 2.f * lr);
    }
    return ok && cudaGetLastError() == cudaSuccess ? FBQ_OK : FBQ_ERR_CUDA;
}

}  // namespace fbq

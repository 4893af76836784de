// Prefill kernel (M > 16) of the FBQuant linear, sm_100a: tcgen05 MMAs with the
// accumulator in tensor memory.
//
//   y = x.dequant(Q,s,z)^T + (x.A^T).B^T        (Algorithm 1 step 6 of the paper)
//
// At prefill the layer is a dense contraction, so it runs on the 5th-generation
// tensor cores.  One CTA owns a tile of 128 weight rows x TOK tokens (TOK = 256,
// or 128 for small M) and issues one 128 x TOK x 16 MMA per 16 elements of K:
// the weight tile is the MMA's A operand (its rows become the 128 TMEM lanes),
// the token tile the B operand (TOK fp32 columns).  Dequantising a weight tile
// once per 256 tokens halves the unpack work per flop against a 128-token tile,
// and the single wide MMA reads 96 bytes of shared memory per cycle, not 128.
//
// Every global read of the K loop is a TMA tensor copy (no multicast), so the
// load/store units only see shared memory:
//   * the token tile of a K block (64 elements of K) lands 128-byte swizzled,
//     ready for the MMA;
//   * the packed codes of the tile's 128 rows land, one quantisation group (two K
//     blocks) per copy, in a small ring that runs several groups ahead;
//   * in the sub-branch blocks the rows of B, and in down-projection mode the
//     rows of A, land 128-byte swizzled as the weight operand itself.
// Roles (20 warps):
//   warps 0-15  producers of the weight operand: warps 0-7 take the even groups,
//               warps 8-15 the odd ones; two threads per weight row, 32 codes of
//               each of the group's two K blocks per thread.  A thread reads its
//               words and (s, z) from the ring, dequantises to the activation type
//               (q - z exact by the exponent trick, one rounding in the product
//               with s), re-pairs the values into natural k order and stores them
//               as 128-byte rows in the same 128-byte swizzle the TMA copies use
//               (bank-conflict free for the stores and for the MMA's reads; the
//               no-swizzle core-matrix layout halved the MMA rate).  Afterwards the same warps drain the
//               accumulator: the tile is staged in shared memory and leaves with
//               TMA tensor stores (epilogue).
//   warp 16     one lane issues tcgen05.mma and hands stages back with
//               tcgen05.commit.
//   warp 17     one lane issues the operand-stage copies (token tile; B or A rows).
//   warps 18-19 keep the ring full: one lane issues the copies of packed codes;
//               all lanes read the tile's scales and zero points with 16-byte
//               loads (one per row and eight groups), realign them and write each
//               group's (s, z) words next to its ring slot.
// The low-rank sub-branch is appended as extra K blocks of the same loop
// (Section 4.3 of the paper adds the up-projection into the shared output):
// their token operand is t = x.A^T (fp32 scratch, rounded once to the activation
// type by the producers), their weight operand is B as stored.  t itself comes
// from the SAME launch: the first blocks of the grid run in down-projection mode
// (both operands by TMA, all of K or a K split each, plain fp32 stores to scratch)
// and raise a flag per token tile; the main CTAs look at the flag (bounded) only
// before their sub-branch blocks, at the very end of their K loop.
// All waits are bounded: a wait that runs out raises FBQ_ERR_TIMEOUT in the
// status word and every role falls through to the common exit.
#include <cuda.h>

#include "fbq_common.cuh"
#include "fbq_dequant.cuh"
#include "fbq_maps.h"
#include "fbq_umma.cuh"

namespace fbq {
namespace {
using namespace ptx;

constexpr int kBN = 128;                           // weight rows per CTA tile (MMA M)
constexpr int kBK = 64;                            // K block (one pipeline stage)
constexpr int kStages = 4;                         // operand stages
constexpr int kRing = 4;                           // groups of packed codes in flight
constexpr int kProducers = 512;                    // threads 0..511: producers, then epilogue
constexpr int kHalf = 256;                         // producers per group (two per weight row)
constexpr int kMmaWarp = kProducers / 32, kTmaWarp = kMmaWarp + 1, kRawWarp = kMmaWarp + 2;
constexpr int kPfThreads = kProducers + 128;         // + MMA warp, TMA warp, two ring warps
constexpr uint32_t kWBytes = kBN * kBK * 2u;       // weight operand tile of a stage
constexpr uint32_t kRawSlot = kBN * 64u;           // ring slot: 128 rows x one group of INT4 codes (INT3 uses 48 of 64)
constexpr int kPfCtrBase = 8;                      // first int of the workspace counters used for the t flags
constexpr uint32_t kPfWaitLimit = 1u << 20;
constexpr uint32_t kPfFlagPolls = 1u << 21;        // polls (256 ns apart) of a token tile's t flag: about half a second

struct PrefillParams {
    const __half *scales;     // [N][K/128]
    const __half *zeros;
    float *t32;               // [M][rank] fp32 scratch: written by the t CTAs, read by the main CTAs
    void *y;                  // [M][N]
    int *status;
    int M, N, K, rank;
    int kb_main;              // K / 64
    int kb_slab;              // ceil(rank / 64) (mode 0)
    int n_t;                  // number of t CTAs = token tiles x rank tiles (0 when rank == 0)
    int rt;                   // rank tiles of 128
    int nt;                   // feature tiles of 128
    int *tflag;               // [token tiles] warps of t CTAs that have stored their part (self-clearing)
    int *tdone;               // [token tiles] main CTAs that have consumed t (self-clearing)
    int splitk, splitt;       // K splits of a main tile / of a t tile (1 unless there are few tokens)
    int cols;                 // token columns in use of a tile of 128 (a multiple of 16)
    float *part;              // [tile][split][TOK][128 rows] fp32 partial tiles (splitk > 1)
    int *split_ctr;           // [tile] splits that have stored their partial (self-clearing)
    uint32_t flag_polls;      // looks (256 ns apart) at a token tile's t flag before the wait gives up
    int test_skip_flag;       // test switch: the t CTAs do not raise the flag (the wait for t must run out)
    void *t16;                // [M][rank_pad] t rounded to the activation type, written by the t CTAs and read by the main
                              // CTAs' TMA copies as one more token operand (NULL: t32 and the producers' conversion)
    int rank_pad;             // columns of t16: rank rounded up to whole K blocks of 64 (the padding is zero)
};

// ---------------------------------------------------------------- PTX helpers of this file
// Bounded by looks (each may sleep in hardware) and inline, unlike ptx::mbar_wait: the producers' loop has no call in it.
__device__ __forceinline__ bool wait_looks(uint32_t bar, uint32_t parity)
{
#pragma unroll 1
    for (uint32_t i = 0; i < kPfWaitLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ bool wait_looks_cluster(uint32_t bar, uint32_t parity)     // sees arrivals from the peer CTA
{
#pragma unroll 1
    for (uint32_t i = 0; i < kPfWaitLimit; ++i)
        if (umma::try_wait_cluster(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ bool elect_one()
{
    uint32_t on;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(on));
    return on != 0u;
}
// Shared-memory loads that stay behind the waits before them (the ones in ptx order themselves with other asm only).
__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// --------------------------------------------------------------------- kernel
// Shared-memory map of a CTA (byte offsets from the 1024-byte aligned base)
template <int TOK> struct Smem {
    static constexpr uint32_t kXBytes = (uint32_t)TOK * kBK * 2u;          // token operand tile of a stage
    static constexpr uint32_t kStageBytes = kXBytes + kWBytes;
    static constexpr uint32_t kRingOff = kStages * kStageBytes;
    static constexpr uint32_t kTableOff = kRingOff + kRing * kRawSlot;
    static constexpr uint32_t kBarOff = kTableOff + kRing * kBN * 4u;
    static constexpr uint32_t kNumBars = 2 * kStages + 2 * kRing + 1 + 4 + 2;  // full, empty, ring full, ring empty, done, epilogue, split
    static constexpr uint32_t kTotal = kBarOff + kNumBars * 8u + 16u;
};

// One launch, 1-D grid.  The first n_t CTAs are "t CTAs": CTA (token tile, rank tile) computes
// t = x.A^T for 256 tokens x 128 rank indices over all of K (both operands by TMA) and stores it as
// fp32 to scratch, then raises the token tile's flag.  The other CTAs are main CTAs, one per
// (feature tile, token tile): y tile = x.dequant(W)^T + t.B^T; they look at the flag only before
// their sub-branch blocks, at the very end of the K loop, by which time the t CTAs (lowest block
// indices, so dispatched first, and with no unpacking to do) have long finished.  The wait is
// bounded like all others.  The last main CTA of a token tile to finish clears the flag again.
// xmap: x [M][K], boxes of TOK rows x 64 elements, 128-byte swizzle
// wmap: packed codes [N][words per row], boxes of 128 rows x one group (64-byte swizzle for INT4)
// amap: A [rank][K], boxes of 128 rows x 64 elements, 128-byte swizzle (t CTAs)
// bmap: B [N][rank], boxes of 128 rows x 64 elements, 128-byte swizzle (main CTAs, rank > 0)
// ymap: y [M][N], boxes of TOK/4 rows x 128 elements, no swizzle (stores)
// tmap: t16 [M][rank_pad], boxes like xmap's (main CTAs, rank > 0, one K split of t)
template <int BITS, typename T, int TOK>
__global__ void __launch_bounds__(kPfThreads, 1)
prefill_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap,
               const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
               const __grid_constant__ CUtensorMap ymap, const __grid_constant__ CUtensorMap tmap, const PrefillParams p)
{
    using L = Smem<TOK>;
    constexpr uint32_t kXBytes = L::kXBytes, kStageBytes = L::kStageBytes;
    constexpr int WPG = (BITS == 4) ? 16 : 12;                  // packed words per row and group
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    if (sbase & 1023u) {                                        // swizzle atoms need a 1024-byte aligned base
        if (threadIdx.x == 0) atomicExch(p.status, (int)FBQ_ERR_CUDA);
        return;
    }
    const uint32_t full0 = sbase + L::kBarOff, empty0 = full0 + 8u * kStages, rfull0 = empty0 + 8u * kStages,
                   rempty0 = rfull0 + 8u * kRing, done_bar = rempty0 + 8u * kRing, epi0 = done_bar + 8u,
                   split_bar = epi0 + 32u, split_bar2 = split_bar + 8u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L::kBarOff + L::kNumBars * 8u);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile int *split_last = abort_flag + 1;                  // 1: this CTA adds up the K splits of its tile

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t cols = TOK == 256 ? 256u : (uint32_t)p.cols, xbytes = cols * kBK * 2u;     // token columns that are copied and multiplied
    const bool t_role = (int)blockIdx.x < p.n_t;                // t CTA or main CTA
    // (token tile, feature or rank tile, K split): with few tokens there are few tiles, so K is split over
    // several CTAs per tile (splitk main CTAs whose fp32 partial tiles the last one to finish adds up,
    // splitt t CTAs that each store their own partial t)
    int m_tile, n_tile, split;
    const int S = t_role ? p.splitt : p.splitk;
    {
        int b = t_role ? (int)blockIdx.x : (int)blockIdx.x - p.n_t;
        split = b % S;
        b /= S;
        const int tiles = t_role ? p.rt : p.nt;
        m_tile = b / tiles;
        n_tile = b % tiles;
    }
    const int m0 = m_tile * TOK, n0 = n_tile * kBN;
    const int G_all = p.kb_main >> 1;
    const int g_begin = (int)((long long)split * G_all / S), g_end = (int)((long long)(split + 1) * G_all / S);
    const int kb_begin = 2 * g_begin;                           // first K block of this CTA's range
    const int kb_x = 2 * (g_end - g_begin);                     // blocks [0, kb_x) of the CTA take their tokens from x
    const int nkb = kb_x + ((t_role || split != 0) ? 0 : p.kb_slab);     // the sub-branch blocks go to split 0

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full0 + 8u * i, t_role ? 1 : kHalf / 32 + 1);   // 8 producer warps + the TMA lane
            mbar_init(empty0 + 8u * i, 1);
        }
        for (int i = 0; i < kRing; ++i) {
            mbar_init(rfull0 + 8u * i, 2);                   // the two ring warps
            mbar_init(rempty0 + 8u * i, kHalf / 32);         // a group is consumed by one half of the producers (8 warps)
        }
        mbar_init(done_bar, 1);
        for (int i = 0; i < 4; ++i) mbar_init(epi0 + 8u * i, 128);     // the four warps of a column quarter
        mbar_init(split_bar, kProducers / 32);               // every epilogue warp has stored its partial chunk
        mbar_init(split_bar2, 1);                            // warp 0 has counted the CTA in
        *abort_flag = 0;
        *split_last = 0;
        fence_barrier_init();
    }
    if (warp == kMmaWarp) {                  // the MMA warp owns the tensor-memory allocation
        umma::tmem_alloc<1>(smem_u32(tmem_slot), (uint32_t)TOK);
        umma::fence_before();
    }
    if (warp == kTmaWarp && lane == 0) {
        prefetch_tensormap(&xmap);
        if (t_role) {
            prefetch_tensormap(&amap);
        } else {
            if (p.rank > 0) prefetch_tensormap(&bmap);
            if (p.t16) prefetch_tensormap(&tmap);
            prefetch_tensormap(&ymap);
        }
    }
    if (warp == kRawWarp && lane == 0)
        prefetch_tensormap(&wmap);
    __syncthreads();
    umma::fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // Programmatic dependent launch: the CTAs of the launch that follows may take their SMs as soon as ours leave
    // them and run their own set-up above; nothing before this point reads or writes global memory, everything
    // after it waits for the preceding launch to have completed (so no bounded wait below spans that launch).
    // Letting the ring of packed codes and the first two dequantised groups start before the wait was measured
    // and changed nothing (68.8 against 68.9 us per linear of a layer step).
    pdl_launch_dependents();
    pdl_wait();

    if (warp < kMmaWarp) {
        bool dead = false;
        if (!t_role) {
            // =================================================== producers
            // Half h of the warps takes the groups g = h, h+2, ... (K blocks 2g and 2g+1, stages 2h
            // and 2h+1); thread (row r, part) dequantises the codes [32*part, +32) of both blocks.
            const int h = warp >> 3, part = (warp >> 2) & 1, r = tid & 127;
            const bool row_ok = n0 + r < p.N;
            const int groups = kb_x >> 1;
            // this thread's words inside a ring slot: block b holds codes [64b, 64b+64) of the group
            uint32_t roff0, roff1;
            if (BITS == 4) {                                // 64-byte rows, 16-byte chunk c stored at c ^ ((row / 2) % 4)
                const uint32_t sw = (uint32_t)(r >> 1) & 3u;
                roff0 = (uint32_t)r * 64u + ((((uint32_t)part) ^ sw) << 4);
                roff1 = (uint32_t)r * 64u + ((((uint32_t)part + 2u) ^ sw) << 4);
            } else {                                        // 48-byte rows of four 12-byte runs
                roff0 = (uint32_t)r * 48u + (uint32_t)part * 12u;
                roff1 = roff0 + 24u;
            }
            const uint32_t ring0 = sbase + L::kRingOff, table0 = sbase + L::kTableOff + (uint32_t)r * 4u;
            // weight tile rows are 128 bytes (64 elements); the 16-byte chunk c of row r sits at c ^ (r % 8)
            const uint32_t wdst = sbase + kXBytes + (uint32_t)(2 * h) * kStageBytes + (uint32_t)r * 128u;
            const uint32_t wsw = (uint32_t)r & 7u;
            const uint32_t fullb = full0 + 16u * h, emptyb = empty0 + 16u * h;
            uint32_t slot = (uint32_t)h, rphase = 0u, ephase = 0u;
#pragma unroll 1
            for (int g = h; g < groups; g += 2) {
                if (!wait_looks(rfull0 + 8u * slot, rphase)) { dead = true; break; }
                constexpr int NW = (BITS == 4) ? 4 : 3;
                uint32_t w[2][NW];
                const uint32_t rs = ring0 + slot * kRawSlot;
                if (BITS == 4) {
                    const uint4 a = lds128(rs + roff0), b = lds128(rs + roff1);
                    w[0][0] = a.x; w[0][1] = a.y; w[0][2] = a.z; w[0][NW - 1] = a.w;
                    w[1][0] = b.x; w[1][1] = b.y; w[1][2] = b.z; w[1][NW - 1] = b.w;
                } else {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        w[0][c] = lds32(rs + roff0 + 4u * c);
                        w[1][c] = lds32(rs + roff1 + 4u * c);
                    }
                }
                const uint32_t sz = lds32(table0 + slot * (kBN * 4u));      // s | z << 16 of (row, group)
                __syncwarp();
                if (lane == 0) mbar_arrive(rempty0 + 8u * slot);   // the warp's words are in registers: the slot may be refilled
                slot += 2u;
                if (slot >= (uint32_t)kRing) { slot -= (uint32_t)kRing; rphase ^= 1u; }
                const float sc = __half2float(__ushort_as_half((unsigned short)(sz & 0xFFFFu)));
                const float ze = __half2float(__ushort_as_half((unsigned short)(sz >> 16)));
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    if (g >= 2 && !wait_looks(emptyb + 8u * b, ephase)) { dead = true; break; }
                    uint32_t wb[16];
                    if (row_ok) {
                        uint32_t d[16];
                        Dequant<BITS, T>::run(w[b], sc, ze, d);
                        natural_pairs<BITS>(d, wb);
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; ++c) wb[c] = 0u;
                    }
#pragma unroll
                    for (int kc = 0; kc < 4; ++kc)
                        sts128(wdst + (uint32_t)b * kStageBytes + ((((uint32_t)(4 * part + kc)) ^ wsw) << 4), wb[4 * kc], wb[4 * kc + 1], wb[4 * kc + 2],
                               wb[4 * kc + 3]);
                }
                if (dead) break;
                fence_proxy_async();                     // generic-proxy stores -> visible to the MMA's reads
                __syncwarp();
                if (lane == 0) {                            // one arrival per warp and block
                    mbar_arrive(fullb);
                    mbar_arrive(fullb + 8u);
                }
                if (g >= 2) ephase ^= 1u;
            }
            // ---- sub-branch blocks: token operand = t (fp32 scratch, rounded once); B arrives by TMA.
            // The halves take them in turn, one token row per thread.
            bool t_ready = false;
#pragma unroll 1
            for (int i = kb_x + h; i < nkb && !dead; i += 2) {
                const int s = i % kStages;
                if (i >= kStages && !wait_looks(empty0 + 8u * s, (uint32_t)(i / kStages - 1) & 1u)) { dead = true; break; }
                if (p.t16) {                                 // both operands of this block arrive by TMA: nothing to write
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full0 + 8u * s);
                    continue;
                }
                if (!t_ready) {                              // every warp of every t CTA of this token tile has stored its part
                    // (every lane looks for itself, one request per warp: an acquire by one lane would order nothing for the others)
                    const int *flag = p.tflag + m_tile;
                    const int target = 16 * p.rt * p.splitt;
                    int seen = 0;
#pragma unroll 1
                    for (uint32_t spin = 0; spin < p.flag_polls; ++spin) {
                        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
                        if (seen >= target) break;
                        __nanosleep(256);
                    }
                    t_ready = __all_sync(0xffffffffu, seen >= target) != 0;
                    if (!t_ready) { dead = true; break; }
                }
                const int j0 = (i - kb_x) * kBK;
                // eight lanes per token row, eight rank indices each (a row per lane touches a line per lane: 5 us of a call)
                const int c = tid & 7, rank4 = p.rank / 4;
                const bool c_ok = j0 + 8 * c < p.rank;       // rank is a multiple of 8: whole chunks
#pragma unroll 1
                for (int u0 = 0; u0 < TOK; u0 += 128) {
                    const int row0 = u0 + ((tid & (kHalf - 1)) >> 3);
                    const float4 *ts = reinterpret_cast<const float4 *>(p.t32) + (size_t)(m0 + row0) * rank4 + (j0 + 8 * c) / 4;
                    float4 ta[4][2];
#pragma unroll
                    for (int u = 0; u < 4; ++u) ta[u][0] = ta[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                    for (int sp = 0; sp < p.splitt; ++sp) {   // partial t of the K splits, in order
                        float4 pv[4][2];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const bool on = c_ok && m0 + row0 + 32 * u < p.M;
                            pv[u][0] = on ? __ldcg(ts + (size_t)32 * u * rank4) : make_float4(0.f, 0.f, 0.f, 0.f);
                            pv[u][1] = on ? __ldcg(ts + (size_t)32 * u * rank4 + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                ta[u][k].x += pv[u][k].x; ta[u][k].y += pv[u][k].y;
                                ta[u][k].z += pv[u][k].z; ta[u][k].w += pv[u][k].w;
                            }
                        ts += (size_t)p.M * rank4;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int rr = row0 + 32 * u;
                        sts128(sbase + (uint32_t)s * kStageBytes + (uint32_t)rr * 128u + ((((uint32_t)c) ^ ((uint32_t)rr & 7u)) << 4),
                               P2<T>::pack(ta[u][0].x, ta[u][0].y), P2<T>::pack(ta[u][0].z, ta[u][0].w),
                               P2<T>::pack(ta[u][1].x, ta[u][1].y), P2<T>::pack(ta[u][1].z, ta[u][1].w));
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + 8u * s);
            }
            if (dead) {
                *abort_flag = 1;
                atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
            }
        }

        // =================================================== epilogue (same sixteen warps)
        // TMEM lane = weight row of the tile, column = token.  Warp w reads lanes 32*(w%4)..+31
        // (the only ones it may address) and the quarter w/4 of the columns.  Mode 0 stages the
        // tile in shared memory as [token][128 features] (the operand stages are free by now) and
        // each column quarter leaves with one TMA tensor store, which also clips the ragged edges.
        if (!dead && nkb > 0 && wait_looks(done_bar, 0)) {
            umma::fence_after();
            const int q = warp & 3, cg = warp >> 2;
            const int nn = n0 + 32 * q + lane;              // output feature (mode 0) / rank index (mode 1)
            const int c_begin = cg * (TOK / 4);
            if (!t_role && S > 1) {
                // ---- K split over S CTAs (TOK = 128: one 32-column chunk per warp).  Every CTA stores its
                // fp32 partial tile; the CTA that counts in last adds the S partials in split order (the
                // result does not depend on which CTA that is) and is the one that writes y.
                // A lane is a feature, so features are the partial tile's contiguous dimension: a warp's store or load is
                // one line.  (With tokens contiguous it touched 32, and the exchange took most of a short call: 77 tokens
                // 4096 -> 4096 rank 0 22.4 us, now 16.4; rank 128, where t was read a row per lane as well, 30.8 and 20.9.)
                const bool mine = m0 + c_begin < p.M;       // uniform over the four warps of a column quarter
                const size_t slice = (size_t)kBN * TOK;
                float *pt = p.part + ((size_t)(m_tile * p.nt + n_tile) * S) * slice + (size_t)c_begin * kBN + 32 * q + lane;
                uint32_t v[32];
                if (mine) {
                    umma::ld32(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)c_begin, v);
                    umma::wait_ld();
                    float *dst = pt + (size_t)split * slice;
#pragma unroll
                    for (int j = 0; j < 32; ++j) __stcg(dst + j * kBN, __uint_as_float(v[j]));
                }
                __threadfence();
                __syncwarp();
                if (lane == 0) mbar_arrive(split_bar);
                if (warp == 0 && lane == 0) {
                    int last = 0;
                    if (wait_looks(split_bar, 0)) {
                        int *ctr = p.split_ctr + m_tile * p.nt + n_tile;
                        last = (atomicAdd(ctr, 1) == S - 1);
                        if (last) atomicExch(ctr, 0);       // left at zero for the next call
                    } else {
                        atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
                    }
                    *split_last = last;
                    __threadfence_block();
                    mbar_arrive(split_bar2);
                }
                const bool last = wait_looks(split_bar2, 0) && *split_last != 0;
                if (last && mine) {
                    __threadfence();
                    float acc[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) acc[j] = 0.f;
#pragma unroll 1
                    for (int sp = 0; sp < S; ++sp) {
                        const float *src = pt + (size_t)sp * slice;
                        float u[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) u[j] = __ldcg(src + j * kBN);
#pragma unroll
                        for (int j = 0; j < 32; ++j) acc[j] += u[j];
                    }
                    unsigned short *sp16 = reinterpret_cast<unsigned short *>(smem + (size_t)c_begin * (kBN * 2)) + 32 * q + lane;
#pragma unroll
                    for (int j = 0; j < 32; ++j) sp16[j * kBN] = to_bits16<T>(acc[j]);
                    fence_proxy_async();                 // staged tile -> visible to the TMA store
                    mbar_arrive(epi0 + 8u * cg);
                    if (q == 0 && lane == 0) {
                        if (wait_looks(epi0 + 8u * cg, 0)) {
                            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                                         ::"l"(reinterpret_cast<uint64_t>(&ymap)), "r"(n0), "r"(m0 + c_begin),
                                           "r"(sbase + (uint32_t)c_begin * (kBN * 2))
                                         : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        } else {
                            atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
                        }
                    }
                }
            } else if (m0 + c_begin < p.M) {                // uniform over the four warps of a column quarter
#pragma unroll 1
                for (int c = c_begin; c < c_begin + TOK / 4; c += 32) {
                    if (m0 + c >= p.M) break;               // warp-uniform
                    uint32_t v[32];
                    umma::ld32(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)c, v);
                    umma::wait_ld();
                    if (!t_role) {
                        unsigned short *sp = reinterpret_cast<unsigned short *>(smem + (size_t)c * (kBN * 2)) + 32 * q + lane;
#pragma unroll
                        for (int j = 0; j < 32; ++j) sp[j * kBN] = to_bits16<T>(__uint_as_float(v[j]));
                    } else if (p.t16) {
                        if (nn < p.rank_pad) {               // rounded once, here; rows of A beyond the rank are zero fill
                            unsigned short *tp = static_cast<unsigned short *>(p.t16) + (size_t)(m0 + c) * p.rank_pad + nn;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (m0 + c + j < p.M) tp[(size_t)j * p.rank_pad] = to_bits16<T>(__uint_as_float(v[j]));
                        }
                    } else {
                        if (nn < p.rank) {                   // 32 lanes = 32 consecutive rank indices: 128-byte stores
                            float *tp = p.t32 + (size_t)split * p.M * p.rank + (size_t)(m0 + c) * p.rank + nn;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (m0 + c + j < p.M) __stcg(tp + (size_t)j * p.rank, __uint_as_float(v[j]));
                        }
                    }
                }
                if (!t_role) {
                    fence_proxy_async();                 // staged tile -> visible to the TMA store
                    mbar_arrive(epi0 + 8u * cg);
                    if (q == 0 && lane == 0) {
                        if (wait_looks(epi0 + 8u * cg, 0)) {
                            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                                         ::"l"(reinterpret_cast<uint64_t>(&ymap)), "r"(n0), "r"(m0 + c_begin),
                                           "r"(sbase + (uint32_t)c_begin * (kBN * 2))
                                         : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // smem may go once it has been read
                        } else {
                            atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
                        }
                    }
                }
            }
            if (t_role) {
                // this warp's part of t is stored: make it visible (to the main CTAs' TMA copies as well), then count the warp in
                asm volatile("fence.proxy.async;" ::: "memory");
                __threadfence();
                __syncwarp();
                if (lane == 0 && !p.test_skip_flag) atomicAdd(p.tflag + m_tile, 1);
            } else if (p.rank > 0 && tid == 0 && split == 0) {
                // this CTA has consumed t (its MMAs are complete).  The last main CTA of the token
                // tile leaves the flag and the count at zero for the next call.
                if (atomicAdd(p.tdone + m_tile, 1) == p.nt - 1) {
                    atomicExch(p.tflag + m_tile, 0);
                    atomicExch(p.tdone + m_tile, 0);
                }
            }
        }
        umma::fence_before();
    } else if (warp == kMmaWarp) {
        // =================================================== MMA warp
        const uint32_t idesc = (1u << 4) | (P2<T>::kFmt << 7) | (P2<T>::kFmt << 10) | ((uint32_t)(cols >> 3) << 17) |
                                   ((uint32_t)(kBN >> 4) << 24);
        // The whole warp walks the loop and one elected lane issues: the MMAs' operands stay in uniform registers.  Under
        // `lane == 0` each was moved there first, 390 cycles per block for four MMAs, and the producers waited for it
        // (18944 x 8192 at 77 tokens 56.2 us, now 50.4; 4096 -> 4096 at 1000 tokens 37.3 and 36.9).
        bool dead = false;
        // descriptors of stage 0; a stage further on is kStageBytes / 16 in their address field
        const uint64_t xd0 = umma::desc_k128(sbase), wd0 = umma::desc_k128(sbase + kXBytes);
        uint32_t s = 0, ph = 0;
#pragma unroll 1
        for (int i = 0; i < nkb; ++i) {
            if (!wait_looks(full0 + 8u * s, ph) || *abort_flag) dead = true;
            if (__any_sync(0xffffffffu, dead)) {
                dead = true;
                break;
            }
            umma::fence_after();
            if (elect_one()) {
                const uint64_t xd = xd0 + s * (kStageBytes >> 4), wd = wd0 + s * (kStageBytes >> 4);
                // every operand tile is K-major with 128-byte rows and the 128-byte swizzle, whether it
                // arrived by TMA or was written by the producers: 32 bytes per 16 elements of K inside a row
#pragma unroll
                for (int j = 0; j < kBK / 16; ++j) umma::mma(tmem_base, wd + 2u * j, xd + 2u * j, idesc, (i > 0 || j > 0) ? 1u : 0u);
                umma::commit(empty0 + 8u * s);                  // stage is free once these MMAs have read it
                if (i == nkb - 1) umma::commit(done_bar);       // accumulator complete
            }
            __syncwarp();
            if (++s == (uint32_t)kStages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (dead && lane == 0) {
            *abort_flag = 1;
            atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
        }
        __syncwarp();
        umma::fence_before();
    } else if (warp == kTmaWarp) {
        // =================================================== operand-stage copies
        if (lane == 0) {
            bool dead = false;
#pragma unroll 1
            for (int i = 0; i < nkb; ++i) {
                const int kb = i, s = i % kStages;
                if ((i >= kStages && !wait_looks(empty0 + 8u * s, (uint32_t)(i / kStages - 1) & 1u)) || *abort_flag) {
                    dead = true;
                    break;
                }
                const uint32_t bar = full0 + 8u * s;
                const uint32_t xt = sbase + (uint32_t)s * kStageBytes, wt = xt + kXBytes;
                if (t_role) {
                    mbar_expect_tx(bar, xbytes + kWBytes);
                    tma_load_2d(xt, &xmap, (kb_begin + kb) * kBK, m0, bar);
                    tma_load_2d(wt, &amap, (kb_begin + kb) * kBK, n0, bar);      // rows of A
                } else if (kb < kb_x) {
                    mbar_expect_tx(bar, xbytes);
                    tma_load_2d(xt, &xmap, (kb_begin + kb) * kBK, m0, bar);
                } else if (p.t16) {
                    if (kb == kb_x) {                        // every warp of every t CTA of this token tile has stored its part
                        const int *flag = p.tflag + m_tile;
                        const int target = 16 * p.rt * p.splitt;
                        int seen = 0;
#pragma unroll 1
                        for (uint32_t spin = 0; spin < p.flag_polls; ++spin) {
                            asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
                            if (seen >= target) break;
                            __nanosleep(256);
                        }
                        if (seen < target) {
                            dead = true;
                            break;
                        }
                        asm volatile("fence.proxy.async;" ::: "memory");
                    }
                    mbar_expect_tx(bar, xbytes + kWBytes);
                    tma_load_2d(xt, &tmap, (kb - kb_x) * kBK, m0, bar);   // t as the token operand
                    tma_load_2d(wt, &bmap, (kb - kb_x) * kBK, n0, bar);   // rows of B
                } else {
                    mbar_expect_tx(bar, kWBytes);
                    tma_load_2d(wt, &bmap, (kb - kb_x) * kBK, n0, bar);   // rows of B
                }
            }
            if (dead) {
                *abort_flag = 1;
                atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
                for (int i = 0; i < 64; ++i) __nanosleep(1000);   // let the copies in flight land before the CTA exits
            }
        }
        __syncwarp();
    } else if (!t_role) {
        // =================================================== ring of packed codes and (s, z) table
        // Two warps; lane l of ring warp v owns the tile rows 64v + l and 64v + l + 32.  Per chunk of
        // eight groups it reads the rows' scales and zero points with 16-byte loads (two aligned chunks of the flat row-major arrays
        // cover any eight consecutive values), realigns them in registers, and before each group's
        // copy writes that group's (s | z << 16) words next to the ring slot.
        const int G = p.K / kGroupFast, groups = kb_x >> 1;     // all groups of a row; groups of this CTA's K range
        const size_t n_chunks = (size_t)p.N * G / 8;        // N is a multiple of 8
        const uint4 *s_arr = reinterpret_cast<const uint4 *>(p.scales), *z_arr = reinterpret_cast<const uint4 *>(p.zeros);
        const int v = warp - kRawWarp;
        size_t a0[2];                                       // aligned 16-byte chunk holding group 0 of the row
        uint32_t off[2];                                    // position of group 0 inside that chunk (0..7)
        bool ok[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int n = n0 + 64 * v + lane + 32 * k;
            ok[k] = n < p.N;
            const size_t f = (size_t)(ok[k] ? n : 0) * G + g_begin;      // first group of this CTA's range
            a0[k] = f >> 3;
            off[k] = (uint32_t)f & 7u;
        }
        uint4 raw[2][2][2];                                 // [row][s|z][low|high chunk] of the next eight groups
        auto fetch = [&](int c) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const size_t a = a0[k] + (size_t)c;
                const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                raw[k][0][0] = (ok[k] && a < n_chunks) ? __ldg(s_arr + a) : zero;
                raw[k][1][0] = (ok[k] && a < n_chunks) ? __ldg(z_arr + a) : zero;
                raw[k][0][1] = (ok[k] && a + 1 < n_chunks) ? __ldg(s_arr + a + 1) : zero;
                raw[k][1][1] = (ok[k] && a + 1 < n_chunks) ? __ldg(z_arr + a + 1) : zero;
            }
        };
        // eight consecutive fp16 values starting `o` values into the 16-value window (lo, hi), as 4 pair-words
        auto realign = [](const uint4 &lo, const uint4 &hi, uint32_t o, uint32_t (&out)[4]) {
            uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            if (o & 2u) {
#pragma unroll
                for (int i = 0; i < 7; ++i) w[i] = w[i + 1];
            }
            if (o & 4u) {
#pragma unroll
                for (int i = 0; i < 5; ++i) w[i] = w[i + 2];
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) out[t] = __funnelshift_r(w[t], w[t + 1], (o & 1u) * 16u);
        };
        bool dead = false;
        const uint32_t ring0 = sbase + L::kRingOff, table0 = sbase + L::kTableOff + (uint32_t)(64 * v + lane) * 4u;
        fetch(0);
#pragma unroll 1
        for (int c = 0; 8 * c < groups && !dead; ++c) {
            uint32_t sz[2][8];                              // (s | z << 16) of [row][group of this chunk]
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                uint32_t sp[4], zp[4];
                realign(raw[k][0][0], raw[k][0][1], off[k], sp);
                realign(raw[k][1][0], raw[k][1][1], off[k], zp);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    sz[k][2 * t] = pf_prmt(sp[t], zp[t], 0x5410u);
                    sz[k][2 * t + 1] = pf_prmt(sp[t], zp[t], 0x7632u);
                }
            }
            if (8 * (c + 1) < groups) fetch(c + 1);
#pragma unroll
            for (int g8 = 0; g8 < 8; ++g8) {
                const int gi = 8 * c + g8;
                if (gi < groups && !dead) {
                    const uint32_t slot = (uint32_t)gi % kRing;
                    if (lane == 0 && ((gi >= kRing && !wait_looks(rempty0 + 8u * slot, (uint32_t)(gi / kRing - 1) & 1u)) || *abort_flag))
                        dead = true;
                    dead = __shfl_sync(0xffffffffu, (int)dead, 0) != 0;     // also orders the table writes after the wait
                    if (!dead) {
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(table0 + slot * (kBN * 4u) + 128u * k), "r"(sz[k][g8]) : "memory");
                        __syncwarp();
                        if (lane == 0) {
                            if (v == 0) {
                                mbar_expect_tx(rfull0 + 8u * slot, (uint32_t)kBN * WPG * 4u);
                                tma_load_2d(ring0 + slot * kRawSlot, &wmap, (g_begin + gi) * WPG, n0, rfull0 + 8u * slot);
                            } else {
                                mbar_arrive(rfull0 + 8u * slot);
                            }
                        }
                    }
                }
            }
        }
        if (dead && lane == 0) {
            *abort_flag = 1;
            atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
            for (int i = 0; i < 64; ++i) __nanosleep(1000);
        }
        __syncwarp();
    }
    __syncthreads();
    if (warp == kMmaWarp) {
        umma::fence_after();
        umma::tmem_free<1>(tmem_base, (uint32_t)TOK);
    }
}

// ---------------------------------------------------------------- CTA-pair variant
// Two CTAs of a cluster (two SMs) share one MMA of 256 weight rows x 256 tokens x 16
// (tcgen05 cta_group::2): each CTA dequantises its own 128 weight rows and stages only HALF of
// the token tile (128 tokens); the tensor cores of both SMs read both halves.  Per CTA and K
// block that is 16 KB less written by TMA and 16 KB less read by the MMA than in the single-CTA
// kernel, and it leaves room for six stages.  MEASURED SLOWER than the single-CTA kernel on B200
// (M = 1024, 4096 -> 4096, INT4, bf16: 47.8 us against 39.8 us; 1120 against 880 cycles per K
// block; with dequantisation, copies and MMAs all switched off the bare hand-shake still takes 760
// cycles per block: the round trip peer arrival -> leader -> multicast commit -> peer is about
// 4500 cycles, more than six stages of MMA time cover), so it is off by default ("prefill_pair"
// option) and kept as a checked alternative.
// The leader CTA (cluster rank 0) issues every MMA; all arrivals that say "stage full" (the
// producer warps of both CTAs, the byte counts of both CTAs' TMA copies) go to the leader's
// barriers; tcgen05.commit with a cluster multicast frees the stage in both CTAs.
constexpr int kPairStages = 6;
struct PairSmem {
    static constexpr uint32_t kXBytes = 128u * kBK * 2u;                   // this CTA's half of the token tile
    static constexpr uint32_t kStageBytes = kXBytes + kWBytes;
    static constexpr uint32_t kRingOff = kPairStages * kStageBytes;
    static constexpr uint32_t kTableOff = kRingOff + kRing * kRawSlot;
    static constexpr uint32_t kBarOff = kTableOff + kRing * kBN * 4u;
    static constexpr uint32_t kNumBars = 2 * kPairStages + 2 * kRing + 1 + 4;
    static constexpr uint32_t kTotal = kBarOff + kNumBars * 8u + 16u;
};
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}

// Grid: 1-D, clusters of two consecutive CTAs.  t CTAs first (pairs: 256 tokens x 256 rank rows),
// then main CTAs (pairs: 256 tokens x 256 features; a padding CTA past the last feature tile
// computes zeros and stores nothing).  Maps as for prefill_kernel, except that the boxes of xmap
// hold 128 token rows.
template <int BITS, typename T>
__global__ void __launch_bounds__(kPfThreads, 1)
prefill_pair_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap,
               const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
               const __grid_constant__ CUtensorMap ymap, const PrefillParams p)
{
    using L = PairSmem;
    constexpr int TOK = 256;                                    // tokens of the pair's tile; this CTA stages 128 of them
    constexpr int kStages = kPairStages;                        // (shadows the single-CTA kernel's depth)
    constexpr uint32_t kXBytes = L::kXBytes, kStageBytes = L::kStageBytes;
    const uint32_t cr = cluster_ctarank();                      // 0: leader (issues the MMAs), 1: peer
    constexpr int WPG = (BITS == 4) ? 16 : 12;                  // packed words per row and group
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    if (sbase & 1023u) {                                        // swizzle atoms need a 1024-byte aligned base
        if (threadIdx.x == 0) atomicExch(p.status, (int)FBQ_ERR_CUDA);
        return;
    }
    const uint32_t full0 = sbase + L::kBarOff, empty0 = full0 + 8u * kStages, rfull0 = empty0 + 8u * kStages,
                   rempty0 = rfull0 + 8u * kRing, done_bar = rempty0 + 8u * kRing, epi0 = done_bar + 8u;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L::kBarOff + L::kNumBars * 8u);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool t_role = (int)blockIdx.x < p.n_t;                // t CTA or main CTA
    int m_tile, n_tile;
    if (t_role) {
        m_tile = (int)blockIdx.x / p.rt;
        n_tile = (int)blockIdx.x % p.rt;                        // tile of rank rows of A
    } else {
        m_tile = ((int)blockIdx.x - p.n_t) / p.nt;
        n_tile = ((int)blockIdx.x - p.n_t) % p.nt;
    }
    const int m0 = m_tile * TOK, n0 = n_tile * kBN;
    const int mh = m0 + 128 * (int)cr;                          // first token of the half this CTA stages
    const int nkb = t_role ? p.kb_main : p.kb_main + p.kb_slab;
    const int kb_x = p.kb_main;                                 // blocks below kb_x take their tokens from x

    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full0 + 8u * i, t_role ? 1 : 17);      // leader's TMA lane + 8 producer warps of each CTA
            mbar_init(empty0 + 8u * i, 1);
        }
        for (int i = 0; i < kRing; ++i) {
            mbar_init(rfull0 + 8u * i, 2);                   // the two ring warps
            mbar_init(rempty0 + 8u * i, kHalf / 32);         // a group is consumed by one half of the producers (8 warps)
        }
        mbar_init(done_bar, 1);
        for (int i = 0; i < 4; ++i) mbar_init(epi0 + 8u * i, 128);     // the four warps of a column quarter
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == kMmaWarp) {                  // the MMA warp owns the tensor-memory allocation
        // the MMA warps of both CTAs of the pair allocate together (same columns in both)
        umma::tmem_alloc<2>(smem_u32(tmem_slot), (uint32_t)TOK);
        umma::fence_before();
    }
    if (warp == kTmaWarp && lane == 0) {
        prefetch_tensormap(&xmap);
        if (t_role) {
            prefetch_tensormap(&amap);
        } else {
            if (p.rank > 0) prefetch_tensormap(&bmap);
            prefetch_tensormap(&ymap);
        }
    }
    if (warp == kRawWarp && lane == 0)
        prefetch_tensormap(&wmap);
    cluster_sync();                          // barriers of both CTAs are initialised before anything arrives on them
    umma::fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp < kMmaWarp) {
        bool dead = false;
        if (!t_role) {
            // =================================================== producers
            // Half h of the warps takes the groups g = h, h+2, ... (K blocks 2g and 2g+1, stages 2h
            // and 2h+1); thread (row r, part) dequantises the codes [32*part, +32) of both blocks.
            const int h = warp >> 3, part = (warp >> 2) & 1, r = tid & 127;
            const bool row_ok = n0 + r < p.N;
            const int groups = p.kb_main >> 1;
            // this thread's words inside a ring slot: block b holds codes [64b, 64b+64) of the group
            uint32_t roff0, roff1;
            if (BITS == 4) {                                // 64-byte rows, 16-byte chunk c stored at c ^ ((row / 2) % 4)
                const uint32_t sw = (uint32_t)(r >> 1) & 3u;
                roff0 = (uint32_t)r * 64u + ((((uint32_t)part) ^ sw) << 4);
                roff1 = (uint32_t)r * 64u + ((((uint32_t)part + 2u) ^ sw) << 4);
            } else {                                        // 48-byte rows of four 12-byte runs
                roff0 = (uint32_t)r * 48u + (uint32_t)part * 12u;
                roff1 = roff0 + 24u;
            }
            const uint32_t ring0 = sbase + L::kRingOff, table0 = sbase + L::kTableOff + (uint32_t)r * 4u;
            // weight tile rows are 128 bytes (64 elements); the 16-byte chunk c of row r sits at c ^ (r % 8)
            const uint32_t wdst = sbase + kXBytes + (uint32_t)r * 128u;
            const uint32_t wsw = (uint32_t)r & 7u;
            const uint32_t lfull0 = mapa_shared(full0, 0);     // the leader's "full" barriers, as seen from this CTA
            uint32_t slot = (uint32_t)h, rphase = 0u;
#pragma unroll 1
            for (int g = h; g < groups; g += 2) {
                if (!wait_looks(rfull0 + 8u * slot, rphase)) { dead = true; break; }
                constexpr int NW = (BITS == 4) ? 4 : 3;
                uint32_t w[2][NW];
                const uint32_t rs = ring0 + slot * kRawSlot;
                if (BITS == 4) {
                    const uint4 a = lds128(rs + roff0), b = lds128(rs + roff1);
                    w[0][0] = a.x; w[0][1] = a.y; w[0][2] = a.z; w[0][NW - 1] = a.w;
                    w[1][0] = b.x; w[1][1] = b.y; w[1][2] = b.z; w[1][NW - 1] = b.w;
                } else {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        w[0][c] = lds32(rs + roff0 + 4u * c);
                        w[1][c] = lds32(rs + roff1 + 4u * c);
                    }
                }
                const uint32_t sz = lds32(table0 + slot * (kBN * 4u));      // s | z << 16 of (row, group)
                __syncwarp();
                if (lane == 0) mbar_arrive(rempty0 + 8u * slot);   // the warp's words are in registers: the slot may be refilled
                slot += 2u;
                if (slot >= (uint32_t)kRing) { slot -= (uint32_t)kRing; rphase ^= 1u; }
                const float sc = __half2float(__ushort_as_half((unsigned short)(sz & 0xFFFFu)));
                const float ze = __half2float(__ushort_as_half((unsigned short)(sz >> 16)));
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int i = 2 * g + b, s = i % kStages;
                    if (i >= kStages && !wait_looks(empty0 + 8u * s, (uint32_t)(i / kStages - 1) & 1u)) { dead = true; break; }
                    uint32_t wb[16];
                    if (row_ok) {
                        uint32_t d[16];
                        Dequant<BITS, T>::run(w[b], sc, ze, d);
                        natural_pairs<BITS>(d, wb);
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; ++c) wb[c] = 0u;
                    }
#pragma unroll
                    for (int kc = 0; kc < 4; ++kc)
                        sts128(wdst + (uint32_t)s * kStageBytes + ((((uint32_t)(4 * part + kc)) ^ wsw) << 4), wb[4 * kc], wb[4 * kc + 1], wb[4 * kc + 2],
                               wb[4 * kc + 3]);
                    fence_proxy_async();                 // generic-proxy stores -> visible to the MMA's reads
                    __syncwarp();
                    if (lane == 0) umma::arrive_cluster(lfull0 + 8u * s);       // one arrival per warp, on the leader's barrier
                }
                if (dead) break;
            }
            // ---- sub-branch blocks: token operand = t (fp32 scratch, rounded once); B arrives by TMA.
            // The halves take them in turn, one token row per thread.
            bool t_ready = false;
#pragma unroll 1
            for (int i = p.kb_main + h; i < nkb && !dead; i += 2) {
                const int s = i % kStages;
                if (i >= kStages && !wait_looks(empty0 + 8u * s, (uint32_t)(i / kStages - 1) & 1u)) { dead = true; break; }
                if (!t_ready) {                              // every warp of every t CTA of this token tile has stored its part
                    // (every lane looks for itself, one request per warp: an acquire by one lane would order nothing for the others)
                    const int *flag = p.tflag + m_tile;
                    const int target = 16 * p.rt;
                    int seen = 0;
#pragma unroll 1
                    for (uint32_t spin = 0; spin < p.flag_polls; ++spin) {
                        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
                        if (seen >= target) break;
                        __nanosleep(256);
                    }
                    t_ready = __all_sync(0xffffffffu, seen >= target) != 0;
                    if (!t_ready) { dead = true; break; }
                }
                const int j0 = (i - p.kb_main) * kBK;
                const int rr = tid & (kHalf - 1);            // token row of this CTA's half of the tile
                if (rr < 128) {
                    const int m = mh + rr;
                    uint32_t xa[32];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        float4 t0 = make_float4(0.f, 0.f, 0.f, 0.f), t1 = t0;
                        if (m < p.M && j0 + 8 * c < p.rank) {              // rank is a multiple of 8: whole chunks
                            const float4 *ts = reinterpret_cast<const float4 *>(p.t32 + (size_t)m * p.rank + j0 + 8 * c);
                            t0 = __ldcg(ts);
                            t1 = __ldcg(ts + 1);
                        }
                        xa[4 * c] = P2<T>::pack(t0.x, t0.y); xa[4 * c + 1] = P2<T>::pack(t0.z, t0.w);
                        xa[4 * c + 2] = P2<T>::pack(t1.x, t1.y); xa[4 * c + 3] = P2<T>::pack(t1.z, t1.w);
                    }
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        sts128(sbase + (uint32_t)s * kStageBytes + (uint32_t)rr * 128u + ((((uint32_t)c) ^ ((uint32_t)rr & 7u)) << 4), xa[4 * c],
                               xa[4 * c + 1], xa[4 * c + 2], xa[4 * c + 3]);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) umma::arrive_cluster(lfull0 + 8u * s);
            }
            if (dead) {
                *abort_flag = 1;
                atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
            }
        }

        // =================================================== epilogue (same sixteen warps)
        // TMEM lane = weight row of the tile, column = token.  Warp w reads lanes 32*(w%4)..+31
        // (the only ones it may address) and the quarter w/4 of the columns.  Mode 0 stages the
        // tile in shared memory as [token][128 features] (the operand stages are free by now) and
        // each column quarter leaves with one TMA tensor store, which also clips the ragged edges.
        if (!dead && nkb > 0 && wait_looks(done_bar, 0)) {
            umma::fence_after();
            const int q = warp & 3, cg = warp >> 2;
            const int nn = n0 + 32 * q + lane;              // output feature (mode 0) / rank index (mode 1)
            const int c_begin = cg * (TOK / 4);
            if (m0 + c_begin < p.M) {                       // uniform over the four warps of a column quarter
#pragma unroll 1
                for (int c = c_begin; c < c_begin + TOK / 4; c += 32) {
                    if (m0 + c >= p.M) break;               // warp-uniform
                    uint32_t v[32];
                    umma::ld32(tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)c, v);
                    umma::wait_ld();
                    if (!t_role) {
                        unsigned short *sp = reinterpret_cast<unsigned short *>(smem + (size_t)c * (kBN * 2)) + 32 * q + lane;
#pragma unroll
                        for (int j = 0; j < 32; ++j) sp[j * kBN] = to_bits16<T>(__uint_as_float(v[j]));
                    } else {
                        if (nn < p.rank) {                   // 32 lanes = 32 consecutive rank indices: 128-byte stores
                            float *tp = p.t32 + (size_t)(m0 + c) * p.rank + nn;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (m0 + c + j < p.M) __stcg(tp + (size_t)j * p.rank, __uint_as_float(v[j]));
                        }
                    }
                }
                if (!t_role) {
                    fence_proxy_async();                 // staged tile -> visible to the TMA store
                    mbar_arrive(epi0 + 8u * cg);
                    if (q == 0 && lane == 0 && n0 < p.N) {   // (a padding CTA past the last feature tile stores nothing)
                        if (wait_looks(epi0 + 8u * cg, 0)) {
                            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                                         ::"l"(reinterpret_cast<uint64_t>(&ymap)), "r"(n0), "r"(m0 + c_begin),
                                           "r"(sbase + (uint32_t)c_begin * (kBN * 2))
                                         : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // smem may go once it has been read
                        } else {
                            atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
                        }
                    }
                }
            }
            if (t_role) {
                // this warp's part of t is stored: make it visible, then count the warp in
                __threadfence();
                __syncwarp();
                if (lane == 0 && !p.test_skip_flag) atomicAdd(p.tflag + m_tile, 1);
            } else if (p.rank > 0 && tid == 0) {
                // this CTA has consumed t (its MMAs are complete).  The last main CTA of the token
                // tile leaves the flag and the count at zero for the next call.
                if (atomicAdd(p.tdone + m_tile, 1) == p.nt - 1) {
                    atomicExch(p.tflag + m_tile, 0);
                    atomicExch(p.tdone + m_tile, 0);
                }
            }
        }
        umma::fence_before();
    } else if (warp == kMmaWarp) {
        // =================================================== MMA warp
        // one MMA of the pair: 256 weight rows (128 per CTA) x 256 tokens (128 staged by each CTA) x 16
        constexpr uint32_t idesc = (1u << 4) | (P2<T>::kFmt << 7) | (P2<T>::kFmt << 10) | ((uint32_t)(TOK >> 3) << 17) |
                                   ((uint32_t)((2 * kBN) >> 4) << 24);
        bool dead = false;
#pragma unroll 1
        for (int i = 0; i < nkb && !dead && cr == 0; ++i) {     // only the leader CTA issues
            const int s = i % kStages;
            if (lane == 0) {
                if (!wait_looks_cluster(full0 + 8u * s, (uint32_t)(i / kStages) & 1u) || *abort_flag) {
                    dead = true;
                } else {
                    umma::fence_after();
                    const uint32_t x_base = sbase + (uint32_t)s * kStageBytes, w_base = x_base + kXBytes;
                    // every operand tile is K-major with 128-byte rows and the 128-byte swizzle, whether it
                    // arrived by TMA or was written by the producers: 32 bytes per 16 elements of K inside a row
#pragma unroll
                    for (int j = 0; j < kBK / 16; ++j)
                        umma::mma_pair(tmem_base, umma::desc_k128(w_base + j * 32), umma::desc_k128(x_base + j * 32), idesc, (i > 0 || j > 0) ? 1u : 0u);
                    umma::commit_pair(empty0 + 8u * s);         // the stage is free, in both CTAs, once these MMAs have read it
                }
            }
            dead = __shfl_sync(0xffffffffu, (int)dead, 0) != 0;
        }
        if (lane == 0) {
            if (dead) {
                *abort_flag = 1;
                atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
            } else if (nkb > 0 && cr == 0) {
                umma::commit_pair(done_bar);                    // accumulators complete in both CTAs
            }
        }
        __syncwarp();
        umma::fence_before();
    } else if (warp == kTmaWarp) {
        // =================================================== operand-stage copies
        if (lane == 0) {
            bool dead = false;
#pragma unroll 1
            for (int i = 0; i < nkb; ++i) {
                const int kb = i, s = i % kStages;
                if ((i >= kStages && !wait_looks(empty0 + 8u * s, (uint32_t)(i / kStages - 1) & 1u)) || *abort_flag) {
                    dead = true;
                    break;
                }
                const uint32_t bar = full0 + 8u * s;
                const uint32_t xt = sbase + (uint32_t)s * kStageBytes, wt = xt + kXBytes;
                // every copy of the pair completes on the LEADER's barrier; the leader announces the bytes of both
                const uint32_t lbar = mapa_shared(bar, 0);
                if (t_role) {
                    if (cr == 0) mbar_expect_tx(bar, 2u * (kXBytes + kWBytes));
                    umma::tma_load_2d_pair(xt, &xmap, kb * kBK, mh, lbar);
                    umma::tma_load_2d_pair(wt, &amap, kb * kBK, n0, lbar);      // rows of A
                } else if (kb < kb_x) {
                    if (cr == 0) mbar_expect_tx(bar, 2u * kXBytes);
                    umma::tma_load_2d_pair(xt, &xmap, kb * kBK, mh, lbar);
                } else {
                    if (cr == 0) mbar_expect_tx(bar, 2u * kWBytes);
                    umma::tma_load_2d_pair(wt, &bmap, (kb - p.kb_main) * kBK, n0, lbar);   // rows of B
                }
            }
            if (dead) {
                *abort_flag = 1;
                atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
                for (int i = 0; i < 64; ++i) __nanosleep(1000);   // let the copies in flight land before the CTA exits
            }
        }
        __syncwarp();
    } else if (!t_role) {
        // =================================================== ring of packed codes and (s, z) table
        // Two warps; lane l of ring warp v owns the tile rows 64v + l and 64v + l + 32.  Per chunk of
        // eight groups it reads the rows' scales and zero points with 16-byte loads (two aligned chunks of the flat row-major arrays
        // cover any eight consecutive values), realigns them in registers, and before each group's
        // copy writes that group's (s | z << 16) words next to the ring slot.
        const int G = p.K / kGroupFast, groups = p.kb_main >> 1;
        const size_t n_chunks = (size_t)p.N * G / 8;        // N is a multiple of 8
        const uint4 *s_arr = reinterpret_cast<const uint4 *>(p.scales), *z_arr = reinterpret_cast<const uint4 *>(p.zeros);
        const int v = warp - kRawWarp;
        size_t a0[2];                                       // aligned 16-byte chunk holding group 0 of the row
        uint32_t off[2];                                    // position of group 0 inside that chunk (0..7)
        bool ok[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int n = n0 + 64 * v + lane + 32 * k;
            ok[k] = n < p.N;
            const size_t f = (size_t)(ok[k] ? n : 0) * G;
            a0[k] = f >> 3;
            off[k] = (uint32_t)f & 7u;
        }
        uint4 raw[2][2][2];                                 // [row][s|z][low|high chunk] of the next eight groups
        auto fetch = [&](int c) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const size_t a = a0[k] + (size_t)c;
                const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                raw[k][0][0] = (ok[k] && a < n_chunks) ? __ldg(s_arr + a) : zero;
                raw[k][1][0] = (ok[k] && a < n_chunks) ? __ldg(z_arr + a) : zero;
                raw[k][0][1] = (ok[k] && a + 1 < n_chunks) ? __ldg(s_arr + a + 1) : zero;
                raw[k][1][1] = (ok[k] && a + 1 < n_chunks) ? __ldg(z_arr + a + 1) : zero;
            }
        };
        // eight consecutive fp16 values starting `o` values into the 16-value window (lo, hi), as 4 pair-words
        auto realign = [](const uint4 &lo, const uint4 &hi, uint32_t o, uint32_t (&out)[4]) {
            uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            if (o & 2u) {
#pragma unroll
                for (int i = 0; i < 7; ++i) w[i] = w[i + 1];
            }
            if (o & 4u) {
#pragma unroll
                for (int i = 0; i < 5; ++i) w[i] = w[i + 2];
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) out[t] = __funnelshift_r(w[t], w[t + 1], (o & 1u) * 16u);
        };
        bool dead = false;
        fetch(0);
        const uint32_t ring0 = sbase + L::kRingOff, table0 = sbase + L::kTableOff + (uint32_t)(64 * v + lane) * 4u;
#pragma unroll 1
        for (int c = 0; 8 * c < groups && !dead; ++c) {
            uint32_t sz[2][8];                              // (s | z << 16) of [row][group of this chunk]
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                uint32_t sp[4], zp[4];
                realign(raw[k][0][0], raw[k][0][1], off[k], sp);
                realign(raw[k][1][0], raw[k][1][1], off[k], zp);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    sz[k][2 * t] = pf_prmt(sp[t], zp[t], 0x5410u);
                    sz[k][2 * t + 1] = pf_prmt(sp[t], zp[t], 0x7632u);
                }
            }
            if (8 * (c + 1) < groups) fetch(c + 1);
#pragma unroll
            for (int g8 = 0; g8 < 8; ++g8) {
                const int gi = 8 * c + g8;
                if (gi < groups && !dead) {
                    const uint32_t slot = (uint32_t)gi % kRing;
                    if (lane == 0 && ((gi >= kRing && !wait_looks(rempty0 + 8u * slot, (uint32_t)(gi / kRing - 1) & 1u)) || *abort_flag))
                        dead = true;
                    dead = __shfl_sync(0xffffffffu, (int)dead, 0) != 0;     // also orders the table writes after the wait
                    if (!dead) {
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(table0 + slot * (kBN * 4u) + 128u * k), "r"(sz[k][g8]) : "memory");
                        __syncwarp();
                        if (lane == 0) {
                            if (v == 0) {
                                mbar_expect_tx(rfull0 + 8u * slot, (uint32_t)kBN * WPG * 4u);
                                tma_load_2d(ring0 + slot * kRawSlot, &wmap, gi * WPG, n0, rfull0 + 8u * slot);
                            } else {
                                mbar_arrive(rfull0 + 8u * slot);
                            }
                        }
                    }
                }
            }
        }
        if (dead && lane == 0) {
            *abort_flag = 1;
            atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
            for (int i = 0; i < 64; ++i) __nanosleep(1000);
        }
        __syncwarp();
    }
    cluster_sync();                          // both CTAs are done with their tensor memory and with each other's barriers
    if (warp == kMmaWarp) {
        umma::fence_after();
        umma::tmem_free<2>(tmem_base, (uint32_t)TOK);
    }
}


int g_pf_pdl = 1;             // launch with programmatic stream serialisation (prefill_set_pdl)

template <int BITS, typename T, int TOK>
cudaError_t launch_kernel(const CUtensorMap &xmap, const CUtensorMap &wmap, const CUtensorMap &amap, const CUtensorMap &bmap,
                          const CUtensorMap &ymap, const CUtensorMap &tmap, const PrefillParams &p, unsigned grid, cudaStream_t s)
{
    auto kern = prefill_kernel<BITS, T, TOK>;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<TOK>::kTotal);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kPfThreads);
    cfg.dynamicSmemBytes = Smem<TOK>::kTotal;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = g_pf_pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, xmap, wmap, amap, bmap, ymap, tmap, p);
}

template <int BITS, typename T>
cudaError_t launch_pair_kernel(const CUtensorMap &xmap, const CUtensorMap &wmap, const CUtensorMap &amap, const CUtensorMap &bmap,
                               const CUtensorMap &ymap, const PrefillParams &p, unsigned grid, cudaStream_t s)
{
    auto kern = prefill_pair_kernel<BITS, T>;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PairSmem::kTotal);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kPfThreads);
    cfg.dynamicSmemBytes = PairSmem::kTotal;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, xmap, wmap, amap, bmap, ymap, p);
}

int g_pair = 0;

// 2-D tensor map of a row-major matrix: `cols` elements per row (16- or 32-bit), `rows` rows,
// boxes of box_cols x box_rows.  Maps of weights are kept (`keep`), those of activations are not.
cudaError_t make_map(CUtensorMap *map, const void *base, bool elem32, size_t cols, size_t rows, int box_cols, int box_rows,
                     CUtensorMapSwizzle swizzle, bool keep)
{
    const MapSpec m = matrix_map(base, elem32 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16, elem32 ? 4 : 2, cols, rows, box_cols,
                                 box_rows, swizzle);
    return keep ? cached_map(map, m) : encode_map(map, m);
}

// K splits of a main tile when all tokens fit one tile of 128: as many as keep the CTA count near the
// number of SMs, at most 8, at least 2 groups of K per split.
int g_pf_skip_flag = 0, g_pf_flag_polls = 0;      // test switches (prefill_set_test)
int g_split_mode = 1;     // 0: never split K, 1: only deep K (>= 8192), 2: whenever tiles are few
int prefill_splits(int N, int K)
{
    if (g_split_mode == 0 || (g_split_mode == 1 && K < 8192)) return 1;
    const int nt = (N + kBN - 1) / kBN, G = K / kGroupFast;
    int s = 148 / nt;
    if (s > 8) s = 8;
    if (s > G / 2) s = G / 2;
    return s < 1 ? 1 : s;
}

template <typename T, int TOK, bool PAIR>
cudaError_t run_prefill(const LinearArgs &a, Workspace &ws, cudaStream_t s, int *launches)
{
    PrefillParams p{};
    p.scales = a.scales;
    p.zeros = a.zeros;
    p.t32 = ws.t_gen;
    p.y = a.y;
    p.status = ws.counters + kCtrStatus;
    p.M = a.M; p.N = a.N; p.K = a.K; p.rank = a.rank;
    p.kb_main = a.K / kBK;
    p.kb_slab = (a.rank + kBK - 1) / kBK;
    const int mt = (a.M + TOK - 1) / TOK;
    // Shared memory is what a block of K waits for (dequantised weights in, operands out): a tile of 128 columns copies
    // and multiplies only those that have tokens.
    p.cols = std::min(TOK, (a.M + 15) / 16 * 16);
    p.nt = (a.N + kBN - 1) / kBN;
    p.rt = (a.rank + kBN - 1) / kBN;
    if (PAIR) {                                     // CTAs come in pairs: feature tiles and rank tiles padded to even counts
        p.nt = (p.nt + 1) & ~1;
        p.rt = (p.rt + 1) & ~1;
    }
    // Few tokens mean few tiles: split K so that about one CTA per SM has work (single-CTA kernel, one
    // token tile).  The same number of splits goes to the t CTAs, which are cheap.
    p.splitk = p.splitt = 1;
    if (!PAIR && TOK == 128 && mt == 1) {             // (the split epilogue is written for one 32-column chunk per warp)
        const int want = prefill_splits(a.N, a.K);
        p.splitk = want;
        p.splitt = (a.rank > 0) ? want : 1;
    }
    p.n_t = mt * p.rt * p.splitt;
    p.tflag = ws.counters + kPfCtrBase;
    p.tdone = p.tflag + mt;
    p.split_ctr = p.tdone + mt;
    p.part = ws.partial;
    p.flag_polls = g_pf_flag_polls > 0 ? (uint32_t)g_pf_flag_polls : kPfFlagPolls;
    p.test_skip_flag = g_pf_skip_flag;
    CUtensorMap xmap, qmap, amap, bmap, ymap;
    cudaError_t e;
    if ((e = make_map(&xmap, a.x, false, (size_t)a.K, (size_t)a.M, kBK, PAIR ? 128 : (TOK == 128 ? p.cols : TOK), CU_TENSOR_MAP_SWIZZLE_128B, false)) != cudaSuccess)
        return e;
    const int wpg = (a.bits == 4) ? 16 : 12;
    if ((e = make_map(&qmap, a.qw, true, (size_t)(a.K / kGroupFast) * wpg, (size_t)a.N, wpg, kBN,
                      a.bits == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE, true)) != cudaSuccess)
        return e;
    if ((e = make_map(&ymap, a.y, false, (size_t)a.N, (size_t)a.M, kBN, TOK / 4, CU_TENSOR_MAP_SWIZZLE_NONE, false)) != cudaSuccess) return e;
    amap = bmap = xmap;
    CUtensorMap tmap = xmap;
    p.t16 = nullptr;
    p.rank_pad = p.kb_slab * kBK;
    if (!PAIR && a.rank > 0 && p.splitt == 1) {
        // t goes from the t CTAs to the main CTAs in the activation type, laid out like x, behind the fp32 slices of t
        p.t16 = ws.t_gen + (((size_t)a.M * a.rank + 3) & ~(size_t)3);
        if ((e = make_map(&tmap, p.t16, false, (size_t)p.rank_pad, (size_t)a.M, kBK, TOK == 128 ? p.cols : TOK, CU_TENSOR_MAP_SWIZZLE_128B, false)) != cudaSuccess) return e;
    }
    if (a.rank > 0) {
        if ((e = make_map(&amap, a.A, false, (size_t)a.K, (size_t)a.rank, kBK, kBN, CU_TENSOR_MAP_SWIZZLE_128B, true)) != cudaSuccess) return e;
        if ((e = make_map(&bmap, a.B, false, (size_t)a.rank, (size_t)a.N, kBK, kBN, CU_TENSOR_MAP_SWIZZLE_128B, true)) != cudaSuccess) return e;
    }
    const unsigned grid = (unsigned)p.n_t + (unsigned)p.nt * (unsigned)mt * (unsigned)p.splitk;
    if (PAIR)
        e = (a.bits == 4) ? launch_pair_kernel<4, T>(xmap, qmap, amap, bmap, ymap, p, grid, s)
                          : launch_pair_kernel<3, T>(xmap, qmap, amap, bmap, ymap, p, grid, s);
    else
        e = (a.bits == 4) ? launch_kernel<4, T, TOK>(xmap, qmap, amap, bmap, ymap, tmap, p, grid, s)
                          : launch_kernel<3, T, TOK>(xmap, qmap, amap, bmap, ymap, tmap, p, grid, s);
    if (e == cudaSuccess) ++*launches;
    return e;
}

inline bool aligned16(const void *q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; }

}  // namespace

// 1: token tiles of 256 run on CTA pairs (cta_group::2); 0: single-CTA kernel
void prefill_set_pair(int on) { g_pair = on ? 1 : 0; }
void prefill_set_split(int mode) { g_split_mode = mode; }
void prefill_set_pdl(int on) { g_pf_pdl = on ? 1 : 0; }
void prefill_set_test(int skip_flag, int flag_polls)
{
    g_pf_skip_flag = skip_flag;
    g_pf_flag_polls = flag_polls;
}

bool prefill_supported(const LinearArgs &a)
{
    return a.group == kGroupFast && a.K % kGroupFast == 0 && a.rank % 8 == 0 && a.rank <= kMaxRank && a.N % 8 == 0 &&
           a.M >= 1 && a.M <= (1 << 22);
}

// Scratch the prefill path needs in the workspace for this call: counters (zero between calls), floats
// of t (one slice per K split), floats of fp32 partial tiles (K split only).
void prefill_workspace_need(const LinearArgs &a, int *counters, size_t *t_floats, size_t *partial_floats)
{
    const int nt = (a.N + kBN - 1) / kBN;
    const int mt128 = (a.M + 127) / 128;
    const int splits = (a.M <= 128) ? prefill_splits(a.N, a.K) : 1;
    *counters = kPfCtrBase + 2 * mt128 + nt * mt128 + 2;
    *t_floats = (size_t)a.M * a.rank * splits + 4 + (size_t)a.M * ((a.rank + 63) / 64 * 64) / 2;      // fp32 slices of t, then t in the activation type
    *partial_floats = (splits > 1) ? (size_t)nt * splits * kBN * 128 : 0;
}

// ws.t_gen must hold M x rank floats and ws.counters prefill_counters_need(M) ints (the caller
// grows them; new counters start at zero and the kernel leaves them at zero).
// Operands that are not 16-byte aligned are refused (the caller then takes the generic kernel).
cudaError_t launch_prefill(const LinearArgs &a, bool dense, Workspace &ws, cudaStream_t s, int *launches)
{
    if (!prefill_supported(a)) return cudaErrorInvalidConfiguration;
    if (!aligned16(a.x) || !aligned16(a.y) || !aligned16(a.qw) || !aligned16(a.scales) || !aligned16(a.zeros) ||
        (a.rank > 0 && (!aligned16(a.A) || !aligned16(a.B))))
        return cudaErrorInvalidConfiguration;
    if (dense) {
        PrefillTuning t;
        t.pdl = g_pf_pdl;
        t.flag_polls = g_pf_flag_polls;
        t.test_skip_flag = g_pf_skip_flag;
        return launch_dense(a, ws, t, s, launches);
    }
    if (a.M <= 128)
        return a.bf16 ? run_prefill<__nv_bfloat16, 128, false>(a, ws, s, launches) : run_prefill<__half, 128, false>(a, ws, s, launches);
    if (g_pair)
        return a.bf16 ? run_prefill<__nv_bfloat16, 256, true>(a, ws, s, launches) : run_prefill<__half, 256, true>(a, ws, s, launches);
    return a.bf16 ? run_prefill<__nv_bfloat16, 256, false>(a, ws, s, launches) : run_prefill<__half, 256, false>(a, ws, s, launches);
}

}  // namespace fbq

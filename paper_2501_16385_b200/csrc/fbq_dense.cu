// Prefill kernel for many tokens, sm_100a: tcgen05 MMAs on CTA pairs over weights that are dequantised once.
//
//   y = x.dequant(Q,s,z)^T + (x.A^T).B^T        (Algorithm 1 step 6 of the paper)
//
// At these sizes the layer is a dense contraction and the tensor cores bound it, if the dequantisation keeps out of
// their way.  Dequantising a weight tile where it is multiplied does it once per token tile (four times at 1024 tokens)
// and every block of K waits for it: the kernel that does so reaches 0.5 of the tensor rate.  Here one persistent launch
// does both halves once: warps that have nothing to do with the MMAs turn the codes into 16-bit weights in a scratch
// matrix W16 (read from L2 mostly: a part of it is written shortly before the tiles in work read it; the whole of it can be
// larger than L2), and the MMA loop is a plain dense one, all of whose operands arrive by TMA.
//
//   warps 8-23   dequantise units of 16 rows x 256 k of W16, claimed from a counter in the order in which the tiles
//                need them (so whichever CTAs are resident do all of them), and tag each finished unit
//   warp 0       operand copies; before the first block of an item it looks at the item's tag (bounded), before the
//                sub-branch blocks at the tags of t
//   warp 1       the leader CTA's lane issues tcgen05.mma.cta_group::2: 256 features x `tok` tokens x 16, K in blocks of 64
//   warp 2       owns the tensor memory; in the leader one lane claims the pair's tiles
//   warp 3       one lane claims the items
//   warps 4-7    epilogue: a tile's accumulator leaves while the next tile's is being made (two in tensor memory)
//
// Features are the MMA's rows (256 per pair), tokens its columns: the token tile can be any multiple of 16 up to 256, so
// it is chosen to fill the last wave of pairs and to waste no columns on a ragged M.  The low-rank branch is
// appended as extra K blocks (Section 4.3 adds the up-projection into the shared output): operands t and B.  t = x.A^T
// comes from tiles of the same loop, the first ones of the launch, rounded once to the activation type.
// Tiles and items are claimed from counters in the order of need, so whoever waits for a t tile or an item waits for a CTA
// that is already resident and itself waits for nobody behind it: any number of resident pairs makes progress, also while
// launches of other streams hold the rest of the SMs.
// Nothing in scratch has to be zero or cleared: tags carry the launch's number, which the last CTA to leave advances.
// All waits are bounded: one that runs out raises FBQ_ERR_TIMEOUT in the status word and every role leaves.
//
// What bounds it: 13824 x 5120 at 4000 tokens takes 440 us (1.3 PFLOP/s, the clock near 1.65 GHz under the power cap; a
// plain cuBLAS GEMM of that size 371 us): 10 us until the first weights are there, 50 us in which the dequantising warps
// take their share of issue slots and L2, then 0.43 us per K block against 0.31 us of MMAs at that clock: the SMs read 32 KB
// each per block from L2.  The weights' operand made in shared memory by each pair (20 KB per block) was measured
// as well: 0.7 us per block, the producers' hand-shake with the other CTA's MMAs is slower than the copies.
#include <cuda.h>

#include <algorithm>

#include "fbq_common.cuh"
#include "fbq_dequant.cuh"
#include "fbq_maps.h"
#include "fbq_umma.cuh"

namespace fbq {
namespace {
using namespace ptx;

constexpr int kBK = 64;                          // K block: 128-byte operand rows
constexpr int kFeat = 256;                       // features of a tile (128 per CTA)
constexpr int kStages = 3, kPer = 2;             // stages of two K blocks: one barrier and one commit for eight MMAs (2 - 6 % over one block)
constexpr uint32_t kHalfBytes = 128u * kBK * 2u; // 128 rows of an operand
constexpr uint32_t kBlockBytes = 2u * kHalfBytes, kStageBytes = kPer * kBlockBytes;
constexpr int kItemK = 256;                      // k extent of a dequantisation item (kFeat rows), which is
constexpr int kUnitRows = 16, kUnits = kFeat / kUnitRows;        // done in units of 16 rows, a warp each,
constexpr int kRowLanes = kItemK / 32, kPassRows = 32 / kRowLanes;   // 32 codes per lane, kPassRows rows at a time
constexpr int kTTok = 128;                       // tokens of a t tile
constexpr int kDqWarp = 8, kDqWarps = 16, kThreads = (kDqWarp + kDqWarps) * 32;
constexpr int kClaims = 4;                       // items claimed ahead
constexpr int kTiles = 8;                        // ring of claimed tiles (see claim_tiles)
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kYBytes = 32u * 128u * 2u;    // staged part of an output tile: 32 tokens x 128 features
constexpr uint32_t kYOff = kStages * kStageBytes;
constexpr uint32_t kBarOff = kYOff + 4u * kYBytes;
constexpr uint32_t kNumBars = 2 * kStages + 4 + 2 * kClaims + kTiles + 1;   // full, empty, accumulator full and free, claims full and taken, tiles, next tile wanted
static_assert(kTiles >= kStages + 2 + 3, "a slot of the tile ring must have been read when it is written again");
constexpr size_t kSmem = kBarOff + kNumBars * 8u + (2 + kClaims + kTiles) * 4u;
// words of the tag scratch: launch number, CTAs that have left, next item, next tile; then tags of items and of t tiles
constexpr int kTagEpoch = 0, kTagDone = 1, kTagNext = 2, kTagTile = 3, kTagFirst = 4;

struct DenseParams {
    const void *x;
    const uint32_t *qw;
    const __half *scales, *zeros;
    void *w16;                // [N][K]
    void *t16;                // [M][rank_pad]
    void *y;                  // [M][N]
    uint32_t *tags;           // see above; unit u of item (ft, kc) at (ft nkc + kc) kUnits + u, CTA c of t tile i at units + 2 i + c
    int *status;
    int M, N, K, rank_pad;
    int nft, ntt, tok;        // feature tiles, token tiles, tokens per tile
    int n_t;                  // t tiles (0 without a sub-branch)
    int rank, a_rows;         // rows of A that a CTA of a t tile loads
    int nkc;                  // items along K
    int wave_ft;              // feature tiles that are in work at the same time
    uint32_t wait_looks;      // 0: waits for tags end by time; else after this many looks
    int test_skip_flag;       // test switch: the t tiles do not tag themselves
};

__device__ __forceinline__ void store_release(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t load_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Four tags, 16-byte aligned.
__device__ __forceinline__ bool tags_are(const uint32_t *p, uint32_t tag)
{
    uint32_t a, b, c, d;
    asm volatile("ld.acquire.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "l"(p) : "memory");
    return ((a ^ tag) | (b ^ tag) | (c ^ tag) | (d ^ tag)) == 0u;
}
__device__ __forceinline__ void store_v8(void *p, const uint32_t *v)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),
                 "r"(v[6]), "r"(v[7])
                 : "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, uint32_t src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(c0), "r"(c1), "r"(src) : "memory");
}

// Whole warp: every lane looks (`there`, an acquiring load) until the first `group` lanes see what they wait for; returns how
// many whole groups of lanes do from there on, or 0 when the bound is hit.  Votes order no memory: the warp barrier carries
// what the lanes have acquired to the one lane that issues the copies.
template <typename F> __device__ __forceinline__ int wait_tags(const DenseParams &p, F there, int group, volatile int *quit)
{
    const unsigned long long t0 = global_ns();
#pragma unroll 1
    for (uint32_t look = 1;; ++look) {
        const unsigned missing = ~__ballot_sync(0xffffffffu, there());
        const int n = (missing ? __ffs(missing) - 1 : 32) / group;
        if (n) {
            __syncwarp();
            return n;
        }
        const bool end = *quit || (p.wait_looks && look >= p.wait_looks) || ((look & 63u) == 0u && global_ns() - t0 > kWaitNs);
        if (__any_sync(0xffffffffu, end)) return 0;
        __nanosleep(32);
    }
}

// Whole warp: brings this CTA's share of `bytes` at `base` (16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_share(const void *base, size_t bytes)
{
    const size_t share = (bytes / gridDim.x + 15) & ~(size_t)15, begin = min(bytes & ~(size_t)15, share * blockIdx.x),
                 end = min(bytes & ~(size_t)15, begin + share);
    constexpr uint32_t kChunk = 4096;
    for (size_t at = begin + (size_t)(threadIdx.x & 31) * kChunk; at < end; at += 32 * kChunk)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(static_cast<const char *>(base) + at), "r"((uint32_t)min((size_t)kChunk, end - at))
                     : "memory");
}

// Items of W16 are claimed from a counter, in the order in which the tiles need them, by one lane per CTA that runs
// kClaims items ahead of the dequantising warps (a claim by every warp for itself: thousands of atomics on one word, 50 us
// of a 45 M weight matrix).  Slot i % kClaims of the ring holds the i-th item, or one past the last as the end.
__device__ __forceinline__ void claim_items(const DenseParams &p, uint32_t cfull0, uint32_t cempty0, volatile int *ring)
{
    const int n_items = p.nft * p.nkc;
#pragma unroll 1
    for (uint32_t i = 0;; ++i) {
        const int item = min((int)atomicAdd(p.tags + kTagNext, 1u), n_items);
        if (i >= kClaims && !mbar_wait(cempty0 + 8u * (i % kClaims), (i / kClaims - 1u) & 1u)) return;
        ring[i % kClaims] = item;
        mbar_arrive(cfull0 + 8u * (i % kClaims));
        if (item >= n_items) return;
    }
}

// The pair's tiles, t tiles first, are claimed by one lane of the leader and handed to both CTAs: the copying, the issuing
// and the epilogue warps read tile i from slot i % kTiles of their CTA's ring.  Tile i is claimed when the copies of tile
// i - 1 are half issued, which hides the claim and deals the tiles out by need (t tiles one per pair, unless fewer pairs
// than t tiles are resident).  A slot is free by then without asking: the copies of tile i - 2 have been issued, so the
// stages of tile i - 5 have been multiplied (kStages stages, at least one per tile; each needs the copies of both CTAs) and
// the epilogues of both CTAs are through with tile i - 7 (two accumulators); slot i % kTiles held tile i - 8.
__device__ __forceinline__ void claim_tiles(const DenseParams &p, int n_all, uint32_t tfull0, uint32_t want, volatile int *tiles, volatile int *quit)
{
    const uint32_t peer_slots = mapa_shared(smem_u32(const_cast<int *>(tiles)), 1), full_a = mapa_shared(tfull0, 0), full_b = mapa_shared(tfull0, 1);
#pragma unroll 1
    for (uint32_t i = 0;; ++i) {
        if (i > 0 && !umma::wait_cluster(want, (i - 1u) & 1u, quit)) return;
        const uint32_t slot = i % kTiles;
        const int q = min((int)atomicAdd(p.tags + kTagTile, 1u), n_all);
        tiles[slot] = q;
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_slots + 4u * slot), "r"(q) : "memory");
        umma::arrive_cluster(full_a + 8u * slot);
        umma::arrive_cluster(full_b + 8u * slot);
        if (q >= n_all) return;
    }
}
// The pair's i-th tile (n_all and above: there are no more), or -1 when the wait for it is given up.
__device__ __forceinline__ int tile_at(uint32_t i, uint32_t tfull0, const volatile int *tiles, volatile int *quit)
{
    const uint32_t slot = i % kTiles;
    return umma::wait_cluster(tfull0 + 8u * slot, (i / kTiles) & 1u, quit) ? tiles[slot] : -1;
}

// A dequantising warp does its unit (kUnitRows rows x kItemK k) of every item of its CTA.  Alone on its latencies (codes
// from HBM, the arithmetic, the fence behind its stores) it would take 3 us per unit, so the next item's codes are
// requested before this one's are turned.
template <int BITS, typename T>
__device__ __forceinline__ bool dequantise(const DenseParams &p, uint32_t tag, uint32_t cfull0, uint32_t cempty0, volatile int *ring)
{
    const int lane = threadIdx.x & 31;
    const int n_items = p.nft * p.nkc, G = p.K / kGroupFast, wave = p.wave_ft * p.nkc, sub = (threadIdx.x >> 5) - kDqWarp;
    constexpr int NW = (BITS == 4) ? 4 : 3, NP = kUnitRows / kPassRows;
    struct Codes {
        uint32_t w[NP][NW];
        __half s[NP], z[NP];
    };
    // the warp's unit of an item: the tags' word, and this lane's place in it: eight lanes per row, 32 codes each
    auto locate = [&](int item, int &word, int &row, int &k0) {
        const int group = item / wave, fts = min(p.wave_ft, p.nft - group * p.wave_ft), r = item - group * wave;
        const int kc = r / fts, ft = group * p.wave_ft + r % fts;
        word = (ft * p.nkc + kc) * kUnits + sub;
        row = ft * kFeat + sub * kUnitRows + lane / kRowLanes;
        k0 = kc * kItemK + lane % kRowLanes * 32;
    };
    auto load = [&](int item, Codes &c) {
        int word, row, k0;
        locate(item, word, row, k0);
#pragma unroll
        for (int i = 0; i < NP; ++i, row += kPassRows) {
            const bool in = row < p.N && k0 < p.K;
            const uint32_t *src = p.qw + (in ? ((size_t)row * p.K + k0) / 32 * NW : 0);
            const size_t g = in ? (size_t)row * G + k0 / kGroupFast : 0;
            if constexpr (BITS == 4) {
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src));
                c.w[i][0] = v.x; c.w[i][1] = v.y; c.w[i][2] = v.z; c.w[i][3] = v.w;
            } else {
#pragma unroll
                for (int j = 0; j < 3; ++j) c.w[i][j] = __ldg(src + j);
            }
            c.s[i] = p.scales[g];
            c.z[i] = p.zeros[g];
        }
    };
    uint32_t i = 0;
    auto take = [&](int &item) -> bool {
        const uint32_t slot = i % kClaims;
        if (!mbar_wait(cfull0 + 8u * slot, (i / kClaims) & 1u)) return false;
        item = ring[slot];
        __syncwarp();
        if (lane == 0) mbar_arrive(cempty0 + 8u * slot);
        ++i;
        return true;
    };
    // An item is announced when the next one's values are about to be stored: its own stores have landed by then, and the
    // fence does not wait for them.
    auto announce = [&](int word) {
        asm volatile("fence.proxy.async;" ::: "memory");        // W16 is read by TMA
        __threadfence();
        __syncwarp();
        if (lane == 0) store_release(p.tags + kTagFirst + word, tag);
    };
    int cur, next, done = -1;
    if (!take(cur)) return false;
    if (cur >= n_items) return true;
    Codes c;
    load(cur, c);
#pragma unroll 1
    for (;;) {
        if (!take(next)) return false;
        Codes n;
        load(min(next, n_items - 1), n);
        int word, row, k0;
        locate(cur, word, row, k0);
        uint32_t out[NP][16];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            uint32_t d[16];
            Dequant<BITS, T>::run(c.w[j], __half2float(c.s[j]), __half2float(c.z[j]), d);
            natural_pairs<BITS>(d, out[j]);
            if (j == 0 && done >= 0) announce(done);
            if (row + kPassRows * j >= p.N || k0 >= p.K) continue;
            T *dst = static_cast<T *>(p.w16) + (size_t)(row + kPassRows * j) * p.K + k0;
            store_v8(dst, out[j]);
            store_v8(dst + 16, out[j] + 8);
        }
        done = word;
        if (next >= n_items) {
            announce(done);
            return true;
        }
        cur = next;
        c = n;
    }
}

// xmap: x [M][K], boxes of tok / 2 rows; xtmap: boxes of kTTok / 2 rows; wmap: W16 [N][K]; amap: A [rank][K];
// bmap: B [N][rank]; tmap: t16 [M][rank_pad], boxes of tok / 2 rows.  All these boxes are 64 elements wide, operand boxes
// of weights 128 rows (of A a_rows), 128-byte swizzle.  ymap: y [M][N], boxes of 16 rows x 128 elements, no swizzle.
template <int BITS, typename T>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
dense_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap xtmap, const __grid_constant__ CUtensorMap wmap,
             const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap, const __grid_constant__ CUtensorMap tmap,
             const __grid_constant__ CUtensorMap ymap, const DenseParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    const uint32_t full0 = sbase + kBarOff, empty0 = full0 + 8u * kStages, accf0 = empty0 + 8u * kStages, acce0 = accf0 + 16u,
                   cfull0 = acce0 + 16u, cempty0 = cfull0 + 8u * kClaims, tfull0 = cempty0 + 8u * kClaims, want = tfull0 + 8u * kTiles;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kBarOff + kNumBars * 8u);
    volatile int *quit = reinterpret_cast<volatile int *>(tmem_slot + 1), *ring = quit + 1, *tiles = ring + kClaims;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t cr = cluster_ctarank();                       // 0: leader
    const int kbx = p.K / kBK, slab = p.rank_pad / kBK;
    const int n_all = p.n_t + p.nft * p.ntt;
    uint32_t *const t_tags = p.tags + kTagFirst + p.nft * p.nkc * kUnits;

    pdl_launch_dependents();
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full0 + 8u * i, 1);
            mbar_init(empty0 + 8u * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(accf0 + 8u * i, 1);
            mbar_init(acce0 + 8u * i, 8);                        // four epilogue warps of each CTA
        }
        for (int i = 0; i < kClaims; ++i) {
            mbar_init(cfull0 + 8u * i, 1);
            mbar_init(cempty0 + 8u * i, kDqWarps);
        }
        for (int i = 0; i < kTiles; ++i) mbar_init(tfull0 + 8u * i, 1);
        mbar_init(want, 1);
        *quit = 0;
        fence_barrier_init();
    }
    if (warp == 2) umma::tmem_alloc<2>(smem_u32(tmem_slot), kTmemCols);
    if (warp == 0 && lane == 0) {
        prefetch_tensormap(&xmap);
        prefetch_tensormap(&wmap);
        prefetch_tensormap(&ymap);
        if (p.n_t) {
            prefetch_tensormap(&xtmap);
            prefetch_tensormap(&amap);
            prefetch_tensormap(&bmap);
            prefetch_tensormap(&tmap);
        }
    }
    // The first pass over codes and x would otherwise meet HBM's latency at every block: with all stages in flight that is
    // 0.43 us per block of K against 0.27 of MMAs.  (Where they are larger, a small part of the time is spent on first passes.)
    if (warp == 3) {
        const size_t cells = (size_t)p.N * p.K, groups = (size_t)p.N * (p.K / kGroupFast) * 2, x_bytes = (size_t)p.M * p.K * 2;
        if (cells <= (size_t)64 << 20) {
            prefetch_share(p.scales, groups);
            prefetch_share(p.zeros, groups);
            prefetch_share(p.qw, cells / 8 * BITS);
        }
        if (x_bytes <= (size_t)32 << 20) prefetch_share(p.x, x_bytes);        // (L2 is the point of coherence: x may still be written)
    }
    umma::fence_before();
    cluster_arrive();
    cluster_wait();                                              // barriers of both CTAs are there
    umma::fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    const uint32_t tag = load_acquire(p.tags + kTagEpoch) + 1u;
    bool ok = true;

    if (warp == 0) {
        // =================================================== operand copies
        const uint32_t lfull0 = mapa_shared(full0, 0);
        uint32_t s = 0, phase = 1u;                              // parity of the stage's previous use
        bool first = true;
#pragma unroll 1
        for (uint32_t it = 0; ok; ++it) {
            const int q = tile_at(it, tfull0, tiles, quit);
            if (q < 0) ok = false;
            if (!__all_sync(0xffffffffu, q >= 0 && q < n_all)) break;
            const bool t_role = q < p.n_t;
            const int ft = t_role ? 0 : (q - p.n_t) / p.ntt, tt = t_role ? 0 : (q - p.n_t) % p.ntt;
            const int wrow = t_role ? 128 * (int)cr : ft * kFeat + 128 * (int)cr;
            const int xrow = t_role ? q * kTTok + (kTTok / 2) * (int)cr : tt * p.tok + (p.tok >> 1) * (int)cr;
            // a t tile's rows beyond the rank are left out (whatever they hold reaches only rows nobody reads); boxes that
            // are mostly out of bounds are slow
            const bool w_load = !t_role || (int)cr * 128 < p.rank_pad;
            const uint32_t bytes = t_role ? (uint32_t)p.a_rows * (p.rank_pad > 128 ? 2u : 1u) * (kBK * 2u) + kTTok * (kBK * 2u)
                                          : 2u * kHalfBytes + (uint32_t)p.tok * (kBK * 2u);
            const int nkb = t_role ? kbx : kbx + slab;
            const int half_way = nkb / (2 * kPer) * kPer;
            int ready = 0;                                       // items of this feature tile known to be there
#pragma unroll 1
            for (int kb = 0; kb < nkb; kb += kPer) {
                const int nb = min(kPer, nkb - kb);
                if (kb == half_way && cr == 0 && lane == 0) mbar_arrive(want);
                if (!t_role && kb < kbx && kb / (kItemK / kBK) >= ready) {
                    // a lane looks at four of the kUnits / 2 tags of this CTA's rows: sixteen items at a time (a look takes
                    // about as long as the copies run ahead, so there should be few)
                    constexpr int group = kUnits / 2 / 4;
                    const int kc = ready + lane / group;
                    const uint32_t *word = p.tags + kTagFirst + (ft * p.nkc + kc) * kUnits + (int)cr * (kUnits / 2) + lane % group * 4;
                    const int n = wait_tags(p, [&] { return kc < p.nkc && tags_are(word, tag); }, group, quit);
                    if (n == 0) { ok = false; break; }
                    ready += n;
                    if (lane == 0) asm volatile("fence.proxy.async;" ::: "memory");
                }
                if (kb == kbx) {                                 // t of this tile's tokens, from both CTAs of each t tile
                    const int t0 = tt * p.tok / kTTok, t1 = (min(p.M, (tt + 1) * p.tok) + kTTok - 1) / kTTok;
                    for (int i = 2 * t0; i < 2 * t1;) {
                        const int n = wait_tags(p, [&] { return i + lane < 2 * t1 && load_acquire(t_tags + i + lane) == tag; }, 1, quit);
                        if (n == 0) { ok = false; break; }
                        i += n;
                    }
                    if (!ok) break;
                    if (lane == 0) asm volatile("fence.proxy.async;" ::: "memory");
                }
                if (lane == 0 && ok) {
                    if (!first && !umma::wait_cluster(empty0 + 8u * s, phase, quit)) {
                        ok = false;
                    } else {
                        const uint32_t bar = lfull0 + 8u * s;
                        if (cr == 0) mbar_expect_tx(full0 + 8u * s, bytes * nb);
                        const bool is_slab = kb >= kbx;
                        for (int j = 0; j < nb; ++j) {
                            const uint32_t wt = sbase + s * kStageBytes + j * kBlockBytes, xt = wt + kHalfBytes;
                            const int k0 = ((is_slab ? kb - kbx : kb) + j) * kBK;
                            if (w_load) umma::tma_load_2d_pair(wt, t_role ? &amap : is_slab ? &bmap : &wmap, k0, wrow, bar);
                            umma::tma_load_2d_pair(xt, t_role ? &xtmap : is_slab ? &tmap : &xmap, k0, xrow, bar);
                        }
                    }
                }
                if (++s == kStages) { s = 0; phase ^= 1u; first = false; }
            }
            ok = __all_sync(0xffffffffu, ok);
        }
    } else if (warp == 1) {
        // =================================================== MMAs
        if (cr == 0 && lane == 0) {
            uint32_t s = 0, phase = 0, it = 0;
            const uint64_t desc0 = umma::desc_k128(sbase);
#pragma unroll 1
            for (; ok; ++it) {
                const int q = tile_at(it, tfull0, tiles, quit);
                if (q < 0) ok = false;
                if (q < 0 || q >= n_all) break;
                const bool t_role = q < p.n_t;
                const int nkb = t_role ? kbx : kbx + slab;
                const uint32_t idesc = umma::idesc_f16(P2<T>::kFmt, 2 * 128, (uint32_t)(t_role ? kTTok : p.tok));
                const uint32_t buf = it & 1u, d = tmem + buf * 256u;
                if (it >= 2 && !umma::wait_cluster(acce0 + 8u * buf, ((it >> 1) - 1u) & 1u, quit)) { ok = false; break; }
                umma::fence_after();
                bool there = mbar_try_wait(full0 + 8u * s, phase) != 0;
#pragma unroll 1
                for (int kb = 0; kb < nkb; kb += kPer) {
                    if (!there && !umma::wait_cluster(full0 + 8u * s, phase, quit)) { ok = false; break; }
                    umma::fence_after();
                    const uint64_t wd = desc0 + s * (kStageBytes >> 4), xd = wd + (kHalfBytes >> 4);
                    const uint32_t freed = empty0 + 8u * s;
                    if (++s == kStages) { s = 0; phase ^= 1u; }
                    umma::mma_pair(d, wd, xd, idesc, kb ? 1u : 0u);
#pragma unroll
                    for (int j = 1; j < kBK / 16; ++j) umma::mma_pair(d, wd + 2 * j, xd + 2 * j, idesc, 1u);
                    if (kb + 1 < nkb) {
                        const uint64_t w2 = wd + (kBlockBytes >> 4), x2 = xd + (kBlockBytes >> 4);
#pragma unroll
                        for (int j = 0; j < kBK / 16; ++j) umma::mma_pair(d, w2 + 2 * j, x2 + 2 * j, idesc, 1u);
                    }
                    umma::commit_pair(freed);
                    there = mbar_try_wait(full0 + 8u * s, phase) != 0;
                }
                if (ok) umma::commit_pair(accf0 + 8u * buf);
            }
        }
    } else if (warp == 2) {
        if (cr == 0 && lane == 0) claim_tiles(p, n_all, tfull0, want, tiles, quit);
        __syncwarp();
    } else if (warp == 3) {
        if (lane == 0) claim_items(p, cfull0, cempty0, ring);
    } else if (warp >= 4 && warp < kDqWarp) {
        // =================================================== epilogue: lane = feature (rank index), column = token
        const int wq = warp & 3;
        const uint32_t lacce0 = mapa_shared(acce0, 0);
        uint32_t it = 0, staged = 0;
#pragma unroll 1
        for (;; ++it) {
            const int q = tile_at(it, tfull0, tiles, quit);
            if (q < 0) ok = false;
            if (q < 0 || q >= n_all) break;
            const uint32_t buf = it & 1u;
            if (!umma::wait_cluster(accf0 + 8u * buf, (it >> 1) & 1u, quit)) { ok = false; break; }
            umma::fence_after();
            const bool t_role = q < p.n_t;
            const int tt = t_role ? q : (q - p.n_t) % p.ntt, cols = t_role ? kTTok : p.tok;
            const int m0 = tt * cols, m_end = min(p.M, m0 + cols);
            const int n = (t_role ? 0 : (q - p.n_t) / p.ntt * kFeat) + 128 * (int)cr + 32 * wq + lane;
            const uint32_t lanes = tmem + buf * 256u + ((uint32_t)(32 * wq) << 16);
#pragma unroll 1
            for (int c = 0; c < cols; c += 32) {
                uint32_t v[32];
                umma::ld32(lanes + (uint32_t)c, v);
                umma::wait_ld();
                if (c + 32 >= cols) {                            // all of the accumulator is in registers
                    umma::fence_before();
                    __syncwarp();
                    if (lane == 0) umma::arrive_cluster(lacce0 + 8u * buf);
                }
                if (t_role) {
                    if (n < p.rank_pad) {
                        unsigned short *dst = static_cast<unsigned short *>(p.t16) + (size_t)(m0 + c) * p.rank_pad + n;
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (j < m_end - (m0 + c)) dst[(size_t)j * p.rank_pad] = n < p.rank ? to_bits16<T>(__uint_as_float(v[j])) : (unsigned short)0;
                    }
                    continue;
                }
                // 32 tokens x 128 features are staged as rows of features and leave by TMA, 16 tokens at a time (which
                // clips the edges of y): stores straight from the lanes took 9 us of a launch
                const uint32_t at = (staged & 3u) * kYBytes;
                if (tid == 4 * 32) asm volatile("cp.async.bulk.wait_group.read 3;" ::: "memory");
                named_barrier_sync(1, 128);                      // the buffer's last copy has been read
                unsigned short *row = reinterpret_cast<unsigned short *>(smem + kYOff + at) + 32 * wq + lane;
#pragma unroll
                for (int j = 0; j < 32; ++j) row[j * 128] = to_bits16<T>(__uint_as_float(v[j]));
                fence_proxy_async();
                named_barrier_sync(1, 128);
                if (tid == 4 * 32) {
                    const int n_first = n - lane;                // warp 4 holds the CTA's first features
                    if (n_first < p.N && m0 + c < p.M) {
                        tma_store_2d(&ymap, sbase + kYOff + at, n_first, m0 + c);
                        if (c + 16 < cols && m0 + c + 16 < p.M) tma_store_2d(&ymap, sbase + kYOff + at + kYBytes / 2, n_first, m0 + c + 16);
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                ++staged;
            }
            if (t_role) {
                asm volatile("fence.proxy.async;" ::: "memory");  // t16 is read by TMA
                __threadfence();
                named_barrier_sync(1, 128);
                if (tid == 4 * 32 && !p.test_skip_flag) store_release(t_tags + 2 * q + cr, tag);
            }
        }
        if (tid == 4 * 32) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    } else if (warp >= kDqWarp) {
        ok = dequantise<BITS, T>(p, tag, cfull0, cempty0, ring);
    }
    if (!ok) {
        *quit = 1;
        atomicExch(p.status, (int)FBQ_ERR_TIMEOUT);
        for (int i = 0; i < 64; ++i) __nanosleep(1000);          // copies in flight land before the CTA leaves
    }
    umma::fence_before();
    __syncthreads();
    cluster_arrive();
    cluster_wait();                                              // nobody needs the other's barriers or tensor memory any more
    if (warp == 2) {
        umma::fence_after();
        umma::tmem_free<2>(tmem, kTmemCols);
    }
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(p.tags + kTagDone, 1u) == gridDim.x - 1) { // the last CTA: the next launch's tags are other ones
            p.tags[kTagDone] = 0;
            p.tags[kTagNext] = 0;
            p.tags[kTagTile] = 0;
            __threadfence();
            p.tags[kTagEpoch] = tag;
        }
    }
}

// ------------------------------------------------------------------ host side
int pairs_of_device()
{
    static int n = 0;
    if (n == 0) {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
        n = std::max(1, sms / 2);
    }
    return n;
}

// Token tiles: a wave of tiles takes 2 cycles per token column and K element (never less than the copies of the weight
// operand take) plus what a tile costs besides, so among the tile widths that M can be cut into the one with the least
// waves x time is taken; M = 1024 on 43 feature tiles: 5 x 208 (3 waves of 74 pairs) instead of 4 x 256 (3 waves too).
int token_tile(int M, int nft, int kb)
{
    const int pairs = pairs_of_device();
    int best = 256;
    double least = 0;
    for (int n = (M + 255) / 256, last = n + 6; n <= last; ++n) {
        const int tok = ((M + n - 1) / n + 15) / 16 * 16;
        if (tok < 64 && n > 1) break;
        const int ntt = (M + tok - 1) / tok, waves = (nft * ntt + pairs - 1) / pairs;
        const double t = waves * (kb * (double)std::max(2 * tok, 300) + 3000.0);
        if (least == 0 || t < least) {
            least = t;
            best = tok;
        }
    }
    return best;
}

// Feature rows of one launch: W16 stays within kW16Most bytes per stream, so a wider matrix (an output head) goes in launches
// of equal parts, whole tiles each.  Small parts end in more partly filled waves (8192 -> 32000, 500 MB, at 1000 tokens: 495 us
// whole, 600 in two), large ones cost nothing (8192 -> 128256, 2.1 GB, at 1000 and 2000 tokens: 1930 and 3650 us in four, 2200
// and 4100 whole).  0: not even one tile's rows fit.
constexpr size_t kW16Most = (size_t)512 << 20;
int launch_rows(int N, int K)
{
    const size_t most = kW16Most / ((size_t)K * 2) / kFeat * kFeat;
    if (most == 0) return 0;
    const size_t n = (N + most - 1) / most;
    return (int)std::min((size_t)N, ((N + n - 1) / n + kFeat - 1) / kFeat * kFeat);
}

// a: the rows of one launch; y has rows of `pitch` elements.
template <int BITS, typename T>
cudaError_t run(const LinearArgs &a, int pitch, Workspace &ws, const PrefillTuning &tune, cudaStream_t s)
{
    DenseParams p{};
    p.x = a.x; p.qw = a.qw; p.scales = a.scales; p.zeros = a.zeros; p.y = a.y;
    p.w16 = ws.w16;
    p.t16 = ws.t_gen;
    p.tags = ws.tags;
    p.status = ws.counters + kCtrStatus;
    p.M = a.M; p.N = a.N; p.K = a.K;
    p.rank_pad = (a.rank + kBK - 1) / kBK * kBK;
    p.rank = a.rank;
    p.a_rows = std::min(128, p.rank_pad);
    p.nft = (a.N + kFeat - 1) / kFeat;
    p.tok = token_tile(a.M, p.nft, a.K / kBK);
    p.ntt = (a.M + p.tok - 1) / p.tok;
    p.n_t = a.rank > 0 ? (a.M + kTTok - 1) / kTTok : 0;
    p.nkc = (a.K + kItemK - 1) / kItemK;
    const int n_pairs = std::min(pairs_of_device(), p.n_t + p.nft * p.ntt);
    p.wave_ft = std::max(1, std::min(p.nft, (n_pairs + p.ntt - 1) / p.ntt));
    p.wait_looks = tune.flag_polls > 0 ? (uint32_t)tune.flag_polls : 0u;
    p.test_skip_flag = tune.test_skip_flag;
    const CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_UINT16;
    const CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_128B;
    CUtensorMap xmap, xtmap, wmap, amap, bmap, tmap, ymap;
    cudaError_t e;
    MapSpec yspec = matrix_map(a.y, dt, 2, a.N, a.M, 128, 16, CU_TENSOR_MAP_SWIZZLE_NONE);
    yspec.strides[0] = (cuuint64_t)pitch * 2;
    if ((e = encode_map(&ymap, yspec)) != cudaSuccess) return e;
    if ((e = encode_map(&xmap, matrix_map(a.x, dt, 2, a.K, a.M, kBK, p.tok / 2, sw))) != cudaSuccess) return e;
    if ((e = cached_map(&wmap, matrix_map(ws.w16, dt, 2, a.K, a.N, kBK, 128, sw))) != cudaSuccess) return e;
    xtmap = amap = bmap = tmap = xmap;
    if (a.rank > 0) {
        if ((e = encode_map(&xtmap, matrix_map(a.x, dt, 2, a.K, a.M, kBK, kTTok / 2, sw))) != cudaSuccess) return e;
        if ((e = encode_map(&tmap, matrix_map(p.t16, dt, 2, p.rank_pad, a.M, kBK, p.tok / 2, sw))) != cudaSuccess) return e;
        if ((e = cached_map(&amap, matrix_map(a.A, dt, 2, a.K, a.rank, kBK, p.a_rows, sw))) != cudaSuccess) return e;
        if ((e = cached_map(&bmap, matrix_map(a.B, dt, 2, a.rank, a.N, kBK, 128, sw))) != cudaSuccess) return e;
    }
    auto kern = dense_kernel<BITS, T>;
    static bool attr_set = false;
    if (!attr_set) {
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem)) != cudaSuccess) return e;
        attr_set = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(2 * n_pairs));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = tune.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, xmap, xtmap, wmap, amap, bmap, tmap, ymap, p);
}

}  // namespace

// The dense kernel pays where its start (10 us until the first weights are there, while no tensor core works) is spread
// over more than three waves of tiles.  Measured, INT4, rank 64, bf16, us per call, this kernel / the one that dequantises
// per token tile: 1024 tokens 4096 -> 4096 (0.9 waves) 46 / 41, 11008 -> 4096 (0.9) 97 / 94, 4096 -> 11008 (2.9) 100 / 115,
// but a layer whose shapes alternate between the two kernels 512 / 503; 4000 tokens 5120 -> 13824 (11.7) 440 / 530, the
// 13B layer 2460 / 2840.  (Few token tiles move the line: 8192 -> 32000 at 500 tokens, 3.4 waves, 320 / 251.)
bool prefill_dense(const LinearArgs &a)
{
    const int rows = launch_rows(a.N, a.K);
    if (a.M <= 128 || rows == 0) return false;
    const int nft = (rows + kFeat - 1) / kFeat, tok = token_tile(a.M, nft, a.K / kBK);
    return nft * ((a.M + tok - 1) / tok) > 3 * pairs_of_device();
}

void dense_workspace_need(const LinearArgs &a, size_t *w16_bytes, size_t *tags, size_t *t_floats)
{
    const size_t rows = launch_rows(a.N, a.K), nft = (rows + kFeat - 1) / kFeat, nkc = (a.K + kItemK - 1) / kItemK;
    *w16_bytes = rows * a.K * 2;
    *tags = kTagFirst + nft * nkc * kUnits + 2 * ((size_t)(a.M + kTTok - 1) / kTTok) + 32;
    *t_floats = (size_t)a.M * ((a.rank + kBK - 1) / kBK * kBK) / 2 + 4;
}

cudaError_t launch_dense(const LinearArgs &a, Workspace &ws, const PrefillTuning &tune, cudaStream_t s, int *launches)
{
    const int rows = launch_rows(a.N, a.K);
    cudaError_t e = cudaSuccess;
    for (int n0 = 0; n0 < a.N && e == cudaSuccess; n0 += rows) {          // (each makes t anew: rank of `rows` of its operations)
        LinearArgs c = a;
        c.N = std::min(rows, a.N - n0);
        c.qw = a.qw + (size_t)n0 * a.K / 32 * a.bits;
        c.scales = a.scales + (size_t)n0 * (a.K / kGroupFast);
        c.zeros = a.zeros + (size_t)n0 * (a.K / kGroupFast);
        if (a.rank > 0) c.B = static_cast<const uint16_t *>(a.B) + (size_t)n0 * a.rank;
        c.y = static_cast<uint16_t *>(a.y) + n0;
        e = a.bits == 4 ? (a.bf16 ? run<4, __nv_bfloat16>(c, a.N, ws, tune, s) : run<4, __half>(c, a.N, ws, tune, s))
                        : (a.bf16 ? run<3, __nv_bfloat16>(c, a.N, ws, tune, s) : run<3, __half>(c, a.N, ws, tune, s));
        if (e == cudaSuccess) ++*launches;
    }
    return e;
}

}  // namespace fbq

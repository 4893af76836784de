// Linears of a few tokens with K split over the CTAs of a cluster (FBQuant linear, sm_100a).
//
// One launch computes  y = x.dequant(Q,s,z)^T + (x.A^T).B^T  (Algorithm 1 step 6 of the paper; the fusion of
// Section 4.3).  What bounds a launch of this size is not the weight stream but what has to happen one after the
// other between the arrival of x and the last store, and the instructions of sixteen warps in between; the kernel is laid
// out so that each of those steps is short:
//
//   * A cluster of CS CTAs owns a range of 32-row tiles; CTA c of it multiplies slice c of K, so a CTA stages only its slice of
//     x (every CTA of the grid reads its x from L2 at the same moment).
//   * The sixteen warps of a CTA are WK parts of the slice x 16 / WK tiles.  Every warp has a ring of its own for the packed codes,
//     filled by its own asynchronous copies: no producer warp, no barrier that another warp has to pass, no descriptor to fetch
//     (tensor copies cost a launch 0.9 us before their first byte).  Codes, scales, zero points and rows of B are on their way
//     before the kernel waits for the preceding one.
//   * A lane loads the run of x whose fragments it holds (32-byte loads), permutes it in registers and never hands it to another
//     lane; sums over x come out of MMAs.  (A conversion through shared memory took 2.7 us of a launch, this 1.2.)
//   * Partial tiles go straight from registers into the shared memory of the CTA that owns the 16 rows (st.async, which counts
//     on that CTA's barrier) and are added there in a fixed order: nothing through L2, no cluster-wide barrier (0.7 us).
//   * t = x.A^T comes from clusters at the head of the grid that do the same with 16 rows of A each.  Every word of it carries
//     the launch's number, so value and "written" travel together and nothing has to be cleared at the end of a launch.  A main CTA
//     takes t in once, with all its threads, and multiplies it with its rows of B as two TF32 terms (exact to 2^-22, any magnitude).
//
// What is left, 4096 -> 4096 INT4 at eight tokens, rank 0 (6.3 us a launch when these were told apart): 0.9 us until the preceding
// kernel has drained, 1.2 x, 1.6 the multiplications, 0.6 the sums and the store, 2 the start of a CTA (it takes the whole SM, so
// none of it overlaps the preceding launch).  In longer launches what counts is the number of instructions: bf16 4096 -> 11008, four
// tokens, a second round of the multiplications adds 2.3 us to 11.4 (55 clocks of the SM for 32 rows x 128 k; the unpacking alone
// takes 40, LOP3 and shifts run at 64 lanes a clock), without them the launch takes 8.2, without the copies of codes 11.1.  So what
// goes with every stage is kept small: the copies' addresses are carried along instead of computed (`issue`), scales come with as
// many rows per instruction as there are lanes.  These two took 4096 -> 11008 from 12.0 to 11.3 us at four tokens and from 14.7 to
// 13.6 at 16, 5120 -> 13824 from 20.3 to 19.0, two problems 4096 -> 11008 as one launch, four tokens, from 21.7 to 19.9.  Two groups
// of a stage in one block of code, for longer chains side by side: 11.5 and 15.6 for 11.4 and 13.7.
//
// 3 to 16 tokens; one problem, or several problems that run as one launch.
#include <algorithm>
#include <cfloat>
#include <cstring>
#include <type_traits>
#include <unordered_map>

#include "fbq_common.cuh"
#include "fbq_ptx.cuh"
#include "fbq_unpack16.cuh"

namespace fbq {
namespace {
using namespace ptx;

constexpr int kW = 16, kThr = kW * 32;       // warps, threads of a CTA
constexpr int kTWK = 8, kTWR = kW / kTWK;    // of a t CTA: parts of the slice of K x granules of A
constexpr int kRows = 32;                    // weight rows of a tile
constexpr int kMostProblems = 8;
constexpr int kMostStages = 4;
constexpr int kGroupBytes = 2048;            // of a stage of a warp's ring, per group of 32 rows of codes
constexpr int kStageA = 4096;                // of a stage of a t CTA: one group of 16 rows of A
constexpr size_t kSmemAll = 227 * 1024;
constexpr int kOffBar = 0;                   // one barrier per receive buffer
constexpr int kOffDims = 64;
constexpr int kOffOver = 256;                // a word per warp: tokens whose x it could not stage scaled up (stage_x)
constexpr int kOffX = 512;

struct alignas(16) SplitDims {
    const void *x, *A, *B;
    const uint8_t *qw;
    const __half *scales, *zeros;
    void *y;
    unsigned long long *t;                   // words of t, [token][rank]: value, above it the number of the launch
    int N, K, G, rank;
    int tiles, R, PT;                        // tiles of the problem, of a cluster, of a pass
    int first_tc, first_mc;                  // first cluster
    int ngt;                                 // sixteen-row granules of A of a t cluster
    int wk_log2, sg, stages;                 // parts of the slice of K that the warps take; groups of a stage, stages of a warp's ring
    int x_wide;                              // x can be read 32 bytes at a time
    int sc_wide, sc_words, sc_pitch;         // scales come in 4-byte words; words and bytes of a row
    int off_px, off_sc, off_b, off_recv, off_t, off_ring, off_trecv, off_tring, tstages;
};
struct SplitParams {
    int n, M, cs_log2, n_tc, poll_limit, skip_t;
    int first_tc[kMostProblems], first_mc[kMostProblems];
    int *status;
    unsigned long long *epoch;               // 2^32 x the number of launches so far, plus the CTAs of this one that are through
    SplitDims p[kMostProblems];
};
static_assert(kOffDims + sizeof(SplitDims) <= kOffOver && kOffOver + kW * 4 <= kOffX, "");

template <typename T> __device__ __forceinline__ void mma16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    if constexpr (std::is_same_v<T, __half>)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The same, started at (c0, c1) in both rows.
template <typename T> __device__ __forceinline__ void mma16_from(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1, float c0, float c1)
{
    if constexpr (std::is_same_v<T, __half>)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const float (&a)[4], float b0, float b1)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])), "r"(__float_as_uint(a[3])), "r"(__float_as_uint(b0)),
          "r"(__float_as_uint(b1)));
}
// 16 bytes into shared memory of a CTA of the cluster; they count towards the transactions of a barrier there.
__device__ __forceinline__ void st_async_v4(uint32_t caddr, uint32_t cbar, const float (&v)[4])
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(caddr), "r"(cbar), "f"(v[0]), "f"(v[1]),
                 "f"(v[2]), "f"(v[3])
                 : "memory");
}

template <typename T> __device__ __forceinline__ float2 pair_to_float(uint32_t v);
template <> __device__ __forceinline__ float2 pair_to_float<__half>(uint32_t v) { return __half22float2(*reinterpret_cast<const __half2 *>(&v)); }
template <> __device__ __forceinline__ float2 pair_to_float<__nv_bfloat16>(uint32_t v)
{
    return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
}
// The pair times f, rounded once.
template <typename T> __device__ __forceinline__ uint32_t pair_scaled(uint32_t v, float f)
{
    using T2 = typename ActTraits<T>::T2;
    T2 f2;
    f2.x = f2.y = ActTraits<T>::from_float(f);
    const T2 r = __hmul2(*reinterpret_cast<const T2 *>(&v), f2);
    return *reinterpret_cast<const uint32_t *>(&r);
}

// A lane's run of x, 32 consecutive elements, straight from L2 (x may have been written by the kernel before, while this SM
// held older lines in its L1): two 32-byte loads, whole sectors, where x is aligned to that.
__device__ __forceinline__ void load_run(const void *src, bool wide, uint32_t (&e)[16])
{
    const uint32_t *s = static_cast<const uint32_t *>(src);
    if (wide) {
#pragma unroll
        for (int i = 0; i < 16; i += 8)
            asm volatile("ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(e[i]), "=r"(e[i + 1]), "=r"(e[i + 2]), "=r"(e[i + 3]), "=r"(e[i + 4]), "=r"(e[i + 5]), "=r"(e[i + 6]), "=r"(e[i + 7])
                         : "l"(s + i));
    } else {
#pragma unroll
        for (int i = 0; i < 16; i += 4)
            asm volatile("ld.global.cg.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(e[i]), "=r"(e[i + 1]), "=r"(e[i + 2]), "=r"(e[i + 3]) : "l"(s + i));
    }
}
// Codes (c0, c1) of the j-th pair that Unpack16 makes of a run of 32.
template <int BITS> __device__ __forceinline__ constexpr int pair_first(int j) { return BITS == 4 ? 8 * (j / 4) + j % 4 : (j < 15 ? 10 * (j / 5) + j % 5 : 30); }
template <int BITS> __device__ __forceinline__ constexpr int pair_second(int j) { return BITS == 4 ? pair_first<4>(j) + 4 : (j < 15 ? pair_first<3>(j) + 5 : 31); }
template <typename T> __device__ __forceinline__ uint32_t pair_of(float v)
{
    const T x = ActTraits<T>::from_float(v);
    const uint32_t u = *reinterpret_cast<const uint16_t *>(&x);
    return u | u << 16;
}

// x of the groups that this warp multiplies, as MMA column fragments [group][eight tokens][quarter of the run][lane] of 16 bytes.
// Lane (token, t) of a fragment needs the run of 32 elements that codes run t of a weight row meet, so it loads that run itself:
// nothing crosses lanes but what the two warps that share the groups stage for each other.  The unpacker's order and field
// weights are applied to x here; (P, X0) of a token and group, the sums of (MAGIC + 2^p kMid) times the staged x and of x, come out of
// MMAs against such rows and rows of field weights, in the lanes that need them.  Tokens past M repeat the last one.
// The tensor core cuts its sums off towards zero, here 1024 times as large as what is left of them, and columns of x that are
// large are so in every group: what a group's products lose, P has to lose as well.  So P is made by the same MMAs in the same order,
// with codes of kMid, and subtracted at the end.  Relative error of y, INT3, fp16, 13824 inputs, one column of each group 1000 times
// as large as the rest / all x of one sign: 2.3e-4 / 2.8e-4, of which the rounding of y is 2.1e-4.  (Products started from
// -MAGIC sum x, an addition less: 1.2e-3 / 2.5e-4; kMid 0: 2.5e-4 / 1.1e-3, half way between the codes 2.4e-4 / 4.2e-4.)
// Two runs are on their way at a time, and never one too many: every CTA asks L2 for the same lines at the same moment, and a load
// that only repeats another costs a launch 0.3 to 0.45 us (4096 -> 4096, 8 tokens, rank 128: with one 7.95 us, with two 8.4, with
// none 7.6).
// What is staged is up x / 2^p, 2^p the field weight of the code that meets x.  In fp16 x / 2^p would be rounded to multiples of 2^-24, so
// `up` is 2^kUp, the largest field weight: nothing is rounded, and `finish` takes it out of the sums.  |x| of 65520 / up and more comes
// out infinite then, which the sums tell: the return value names the tokens (bit t: token 2t of the eight, bit 4 + t: 2t + 1; the warps of
// a part are a multiple of MT, so that all runs of a lane belong to one).  The part is staged again with up = 1 for these, where
// a rounding of 2^-19 is nothing beside an x of 1000.  (13B layer, 16 tokens, fp16:
// 101.5 us, 99.8 with x / 2^p and no second pass; with small x found by the sum of |x| instead, and staged again scaled up, 103.0.)
template <int BITS> constexpr float kMid = BITS == 4 ? 6.f : 2.f;
// Products start from -P all the same in bf16, whose 128 x cut off is lost in its rounding of y (1.7e-3), from nine tokens on: 16 tokens, rank 64,
// 4096 -> 11008 15.26 -> 14.80 us, 11008 -> 4096 18.3 -> 17.8; with 8 tokens, rank 128, 13824 -> 5120 17.7 -> 18.3.
template <typename T, int MT> constexpr bool kFromP = std::is_same_v<T, __nv_bfloat16> && MT == 2;
template <int BITS, typename T> constexpr int kUp = std::is_same_v<T, __half> ? (BITS == 4 ? 4 : 6) : 0;      // (bf16 has the exponents)
template <int BITS, typename T, int MT>
__device__ __forceinline__ uint32_t stage_x(const T *x, int K, int M, bool wide, uint8_t *xs, float4 *px, int groups, int part, int parts, int lane, float up)
{
    const int n = lane >> 2, t = lane & 3, total = groups * MT;
    bool over0 = false, over1 = false;
    auto load = [&](int it, uint32_t (&e)[16]) {
        const int grp = it / MT, b = it - grp * MT;
        load_run(x + (size_t)min(8 * b + n, M - 1) * K + grp * kGroupFast + 32 * t, wide, e);
    };
    auto convert = [&](int it, const uint32_t (&e)[16]) {
        uint32_t h[16];
        float d[4] = {};
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            constexpr auto div = [](int c) { return Unpack16<BITS, T>::div_log2(c); };
            const int c0 = pair_first<BITS>(j), c1 = pair_second<BITS>(j);
            h[j] = __byte_perm(e[c0 >> 1], e[c1 >> 1], ((c0 & 1) ? 0x32u : 0x10u) | ((c1 & 1) ? 0x7600u : 0x5400u));
            if (kUp<BITS, T> > 0 || div(c0) > 0) h[j] = pair_scaled<T>(h[j], up / (float)(1 << div(c0)));
            if (j & 1) {
                constexpr float magic = Unpack16<BITS, T>::kMagic;
                const float w0 = (float)(1 << div(pair_first<BITS>(j - 1))), w1 = (float)(1 << div(c0));
                mma16<T>(d, pair_of<T>(magic + w0 * kMid<BITS>), pair_of<T>(w0), pair_of<T>(magic + w1 * kMid<BITS>), pair_of<T>(w1), h[j - 1], h[j]);
            }
        }
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4)
            *reinterpret_cast<uint4 *>(xs + (((it * 4 + q4) * 32 + lane) << 4)) = make_uint4(h[4 * q4], h[4 * q4 + 1], h[4 * q4 + 2], h[4 * q4 + 3]);
        if constexpr (kUp<BITS, T> > 0) {
            over0 = over0 || !(fabsf(d[2]) <= FLT_MAX);
            over1 = over1 || !(fabsf(d[3]) <= FLT_MAX);
        }
        if (lane < 4) px[it * 4 + lane] = make_float4(d[0], d[1], d[2], d[3]);
    };
    int it = part;
#pragma unroll 1
    for (; it + parts < total; it += 2 * parts) {
        uint32_t e[2][16];
        load(it, e[0]);
        load(it + parts, e[1]);
        convert(it, e[0]);
        convert(it + parts, e[1]);
    }
    if (it < total) {
        uint32_t e[16];
        load(it, e);
        convert(it, e);
    }
    if constexpr (kUp<BITS, T> > 0) return (__ballot_sync(0xFFFFFFFFu, over0) & 15u) | (__ballot_sync(0xFFFFFFFFu, over1) & 15u) << 4;
    return 0u;
}
// The same for a t CTA: x as it is.
template <typename T, int MT>
__device__ __forceinline__ void stage_x_plain(const T *x, int K, int M, bool wide, uint8_t *xs, int groups, int part, int lane)
{
    const int n = lane >> 2, t = lane & 3, total = groups * MT;
#pragma unroll 1
    for (int it = part; it < total; it += kTWR) {
        const int grp = it / MT, b = it - grp * MT;
        uint32_t e[16];
        load_run(x + (size_t)min(8 * b + n, M - 1) * K + grp * kGroupFast + 32 * t, wide, e);
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4)
            *reinterpret_cast<uint4 *>(xs + (((it * 4 + q4) * 32 + lane) << 4)) = make_uint4(e[4 * q4], e[4 * q4 + 1], e[4 * q4 + 2], e[4 * q4 + 3]);
    }
}

// One quantisation group of a tile: 32 rows x 8 MT tokens.  `codes` = this lane's place in the group's codes.
template <int BITS, typename T, int MT>
__device__ __forceinline__ void multiply_group(const uint8_t *codes, const uint8_t *xg, const uint8_t *pxg, const uint8_t *sc, uint32_t zoff, uint32_t srow8,
                                               float (&acc)[2][MT][4])
{
    constexpr int NW = BITS == 4 ? 4 : 3, GB = BITS == 4 ? 64 : 48;
    uint32_t ha[2][16], hb[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t wa[NW], wb[NW];
        const uint8_t *c = codes + h * 16 * GB;
        if constexpr (BITS == 4) {
            const uint4 a = *reinterpret_cast<const uint4 *>(c), b = *reinterpret_cast<const uint4 *>(c + 8 * GB);
            wa[0] = a.x; wa[1] = a.y; wa[2] = a.z; wa[3] = a.w;
            wb[0] = b.x; wb[1] = b.y; wb[2] = b.z; wb[3] = b.w;
        } else {
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                wa[i] = reinterpret_cast<const uint32_t *>(c)[i];
                wb[i] = reinterpret_cast<const uint32_t *>(c + 8 * GB)[i];
            }
        }
        Unpack16<BITS, T>::run(wa, ha[h]);
        Unpack16<BITS, T>::run(wb, hb[h]);
    }
    float fs[4], fz[4];                                                       // rows g, g + 8, g + 16, g + 24
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        fs[r] = __half2float(*reinterpret_cast<const __half *>(sc + r * srow8));
        fz[r] = kMid<BITS> - __half2float(*reinterpret_cast<const __half *>(sc + r * srow8 + zoff));
    }
    constexpr bool kFrom = kFromP<T, MT>;
    float d[2][MT][4] = {}, p[MT][2], x0[MT][2];
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4)
#pragma unroll
        for (int b = 0; b < MT; ++b) {
            const uint4 xv = *reinterpret_cast<const uint4 *>(xg + (b * 4 + q4) * 512);
            if (q4 == 0) {
                const float4 v = *reinterpret_cast<const float4 *>(pxg + b * 64);     // (P, P, X0, X0) of tokens 8b + 2t, 8b + 2t + 1
                p[b][0] = v.x;
                p[b][1] = v.y;
                x0[b][0] = v.z;
                x0[b][1] = v.w;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (kFrom && q4 == 0) mma16_from<T>(d[h][b], ha[h][4 * q4], hb[h][4 * q4], ha[h][4 * q4 + 1], hb[h][4 * q4 + 1], xv.x, xv.y, -p[b][0], -p[b][1]);
                else mma16<T>(d[h][b], ha[h][4 * q4], hb[h][4 * q4], ha[h][4 * q4 + 1], hb[h][4 * q4 + 1], xv.x, xv.y);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) mma16<T>(d[h][b], ha[h][4 * q4 + 2], hb[h][4 * q4 + 2], ha[h][4 * q4 + 3], hb[h][4 * q4 + 3], xv.z, xv.w);
        }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
#pragma unroll
            for (int b = 0; b < MT; ++b)
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    acc[h][b][2 * r + c] = fmaf(fs[2 * h + r], fmaf(fz[2 * h + r], x0[b][c], kFrom ? d[h][b][2 * r + c] : d[h][b][2 * r + c] - p[b][c]), acc[h][b][2 * r + c]);
        }
}

// This warp's partial sums of 16 rows, to the CTA of the cluster that finishes them: [granule slot][slice, part][eight tokens][lane].
template <int MT>
__device__ __forceinline__ void send_granule(uint32_t recv, uint32_t bar, int gi, int cs_log2, int crank, int wk_log2, int part, int lane, const float (&acc)[MT][4])
{
    const uint32_t owner = (uint32_t)(gi & ((1 << cs_log2) - 1)), slot = (uint32_t)gi >> cs_log2;
    const uint32_t dst = mapa_shared(recv + ((((slot << cs_log2) + crank) << wk_log2) + part) * MT * 512u + lane * 16u, owner), cbar = mapa_shared(bar, owner);
#pragma unroll
    for (int b = 0; b < MT; ++b) st_async_v4(dst + b * 512u, cbar, acc[b]);
}
// Granules of `n` that CTA `crank` finishes.
__device__ __forceinline__ int owned(int n, int cs_log2, int crank) { return (n + (1 << cs_log2) - 1 - crank) >> cs_log2; }

// A word of t: value and number of the launch, an element of 64 bits to both accesses, so that whoever sees the number sees the value.
// (Of the elements of a vector access nothing says that they are seen together.)
__device__ __forceinline__ void store_t(unsigned long long *w, float v, uint32_t tag)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(w), "l"((unsigned long long)tag << 32 | __float_as_uint(v)));
}
__device__ __forceinline__ uint4 load_t2(const unsigned long long *w)        // two of them
{
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(w));
    return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All but the latest n - 1 groups of copies of this thread have arrived.
__device__ __forceinline__ void cp_async_wait_stage(int n)
{
    if (n == kMostStages) asm volatile("cp.async.wait_group 3;" ::: "memory");
    else if (n == 3) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else if (n == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }

// This launch's number, which the words of its t carry: never 0, which words that no launch has written hold and lanes that have
// not looked yet.  It comes round after 2^31 launches; a word still holds the number of that many launches ago only where no call
// since then had as many tokens and ranks, and is written by this launch's t CTA all the same.
__device__ __forceinline__ uint32_t launch_number(const unsigned long long *epoch) { return (uint32_t)(__ldcg(epoch) >> 32) | 0x80000000u; }

template <typename T, int MT>
__device__ __forceinline__ void t_program(const SplitParams &sp, const SplitDims &p, uint8_t *smem, int lc, int crank, int g0, int Gs)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, M = sp.M, K = p.K, rank = p.rank;
    const uint32_t sbase = smem_u32(smem), rbar = sbase + kOffBar;
    const int row0 = lc * p.ngt * 16, ngran = min(p.ngt, (rank - row0 + 15) / 16);
    // this warp's groups of the slice, and granules wr, wr + kTWR, ... of 16 rows of A
    const int wk = warp % kTWK, wr = warp / kTWK, gb = Gs * wk / kTWK, mine = Gs * (wk + 1) / kTWK - gb, total = mine * ((ngran - wr + kTWR - 1) / kTWR);
    const int stages = p.tstages;
    const uint32_t ring = sbase + p.off_tring + (uint32_t)(warp * stages * kStageA);
    // A stage: one group of a granule, rows of 256 bytes whose 16-byte units c lie at c ^ (c >> 3) ^ 2 (row & 1) (within the
    // half row): the fragment reads below meet each bank once
    const int ar = lane >> 4, ac = lane & 15;
    const T *asrc = static_cast<const T *>(p.A) + (size_t)(row0 + ar) * K + (size_t)(g0 + gb) * kGroupFast + ac * 8;
    const uint32_t adst = ring + (uint32_t)(ar * 256 + ((ac & 8) | ((ac & 7) ^ (ac >> 3) ^ (2 * ar))) * 16);
    int issued = 0, ig = 0, igran = wr, islot = 0;
    auto issue = [&]() {
        if (issued < total) {
            const T *src = asrc + (size_t)igran * 16 * K + ig * kGroupFast;
#pragma unroll
            for (int i = 0; i < 8; ++i) cp_async16(adst + islot * kStageA + i * 512, src + (size_t)(2 * i) * K);
            ++issued;
            if (++islot == stages) islot = 0;
            if (++ig == mine) {
                ig = 0;
                igran += kTWR;
            }
        }
        cp_async_commit();
    };
#pragma unroll 1
    for (int i = 0; i < stages; ++i) issue();
    uint8_t *xs = smem + kOffX + (size_t)gb * MT * 2048;
    const T *x = static_cast<const T *>(p.x) + (size_t)(g0 + gb) * kGroupFast;
    const bool wide = p.x_wide != 0;
    unsigned long long *tw = p.t;
    pdl_wait();
    const uint32_t tag = launch_number(sp.epoch);
    stage_x_plain<T, MT>(x, K, M, wide, xs, mine, wr, lane);
    __syncthreads();
    cluster_wait();                                                           // the other CTAs of the cluster have started
    int slot = 0;
#pragma unroll 1
    for (int gran = wr; gran < ngran; gran += kTWR) {
        float acc[MT][4] = {};
#pragma unroll 1
        for (int i = 0; i < mine; ++i) {
            cp_async_wait_stage(stages);
            __syncwarp();
            const uint8_t *a = smem + p.off_tring + (warp * stages + slot) * kStageA + g * 256;
            const uint8_t *xg = xs + (size_t)i * MT * 2048 + lane * 16;
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
                const uint8_t *u = a + (((t >> 1) << 3) | ((4 * (t & 1) + q4) ^ (t >> 1) ^ (2 * (g & 1)))) * 16;
                const uint4 r0 = *reinterpret_cast<const uint4 *>(u), r8 = *reinterpret_cast<const uint4 *>(u + 8 * 256);
#pragma unroll
                for (int b = 0; b < MT; ++b) {
                    const uint4 xv = *reinterpret_cast<const uint4 *>(xg + (b * 4 + q4) * 512);
                    mma16<T>(acc[b], r0.x, r8.x, r0.y, r8.y, xv.x, xv.y);
                    mma16<T>(acc[b], r0.z, r8.z, r0.w, r8.w, xv.z, xv.w);
                }
            }
            __syncwarp();
            issue();
            if (++slot == stages) slot = 0;
        }
        send_granule<MT>(sbase + p.off_trecv, rbar, gran, sp.cs_log2, crank, 3, wk, lane, acc);
    }
    const int cs = 1 << sp.cs_log2;
    if (!mbar_wait(rbar, 0u)) atomicExch(sp.status, (int)FBQ_ERR_TIMEOUT);
#pragma unroll 1
    for (int gran = crank; gran < ngran; gran += cs)
#pragma unroll 1
        for (int e = threadIdx.x; e < MT * 128; e += kThr) {
            const float *src = reinterpret_cast<const float *>(smem + p.off_trecv) + (size_t)(gran >> sp.cs_log2 << sp.cs_log2) * kTWK * MT * 128 + e;
            float v = 0.f;
#pragma unroll 1
            for (int c = 0; c < cs * kTWK; c += kTWK) {
                float w[kTWK];
#pragma unroll
                for (int k = 0; k < kTWK; ++k) w[k] = src[(size_t)(c + k) * MT * 128];
#pragma unroll
                for (int k = 0; k < kTWK; ++k) v += w[k];
            }
            const int l = (e >> 2) & 31, token = (e >> 7) * 8 + 2 * (l & 3) + (e & 1), row = row0 + gran * 16 + (l >> 2) + 8 * ((e >> 1) & 1);
            if (token < M && row < rank && !sp.skip_t) store_t(tw + (size_t)token * rank + row, v, tag);
        }
}

// Returns whether one of this thread's sums is not finite.
template <int BITS, typename T, int MT>
__device__ __forceinline__ bool main_program(const SplitParams &sp, const SplitDims &p, uint8_t *smem, int lc, int crank, int g0, int Gs)
{
    constexpr int GB = BITS == 4 ? 64 : 48, kUnits = GB / 16;                 // bytes of a row and group, 16-byte units
    // (fields that are used past the wait are read here: shared memory would be read again after every barrier)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, M = sp.M, cs_log2 = sp.cs_log2, cs = 1 << cs_log2;
    const int N = p.N, K = p.K, rank = p.rank, PT = p.PT, stages = p.stages;
    const uint32_t sbase = smem_u32(smem), rbar = sbase + kOffBar;
    const int tile0 = lc * p.R, ntiles = min(p.R, p.tiles - tile0), nrow0 = tile0 * kRows, npass = (ntiles + PT - 1) / PT;
    // this warp's groups of the slice and tiles wr, wr + wr_n, ...
    const int wkl = p.wk_log2, wr_n = kW >> wkl, wk = warp & ((1 << wkl) - 1), wr = warp >> wkl, gb = Gs * wk >> wkl, mine = (Gs * (wk + 1) >> wkl) - gb;
    const int my_tiles = ntiles > wr ? (ntiles - wr + wr_n - 1) / wr_n : 0, sg = p.sg, stage_bytes = sg * kGroupBytes;

    // ---- the warp's ring of packed codes: a stage is sg groups of a tile, [group][row][64 or 48 bytes] ----
    const uint32_t ring = sbase + p.off_ring + (uint32_t)(warp * stages * stage_bytes);
    const int row_bytes = p.G * GB;
    // this lane's first row and 16-byte unit of it; the next ones are 32 units on, in rows of `units`
    const int units = sg * kUnits, r0 = sg == 2 ? lane / (2 * kUnits) : lane / kUnits, c0 = lane - r0 * units, rstep = sg == 2 ? 32 / (2 * kUnits) : 32 / kUnits;
    const uint8_t *qsrc = p.qw + (size_t)(g0 + gb) * GB + (size_t)(nrow0 + wr * kRows + r0) * row_bytes + c0 * 16;   // of the stage to come
    const ptrdiff_t qnext = (ptrdiff_t)(wr_n * kRows) * row_bytes - (ptrdiff_t)(mine + sg - 1) / sg * sg * GB;       // end of a tile's stages -> the next tile
    const size_t qstep = (size_t)rstep * row_bytes;
    const uint32_t qdst = ring + (uint32_t)((c0 >= kUnits ? (kRows * GB) - GB : 0) + r0 * GB + c0 * 16), ring_bytes = (uint32_t)(stages * stage_bytes);
    int ptile = mine > 0 ? wr : ntiles, pg = 0;
    uint32_t pat = 0;                                                         // place of the stage in the ring
    auto issue = [&]() {
        if (ptile < ntiles) {
            const uint8_t *src = qsrc;
            const int last = N - 1 - (nrow0 + ptile * kRows);                 // rows past N repeat the last one
            if constexpr (BITS == 4) {
                // unit c0 of rows r0, r0 + rstep, ...
                const uint32_t d = qdst + pat;
                if (last < kRows - 1) {
#pragma unroll 1
                    for (int i = 0; i < units && pg + (c0 >> 2) < mine; ++i) cp_async16(d + i * rstep * GB, src + (ptrdiff_t)(min(r0 + rstep * i, last) - r0) * row_bytes);
                } else if (sg == 2) {
                    if (pg + (c0 >> 2) < mine) {
#pragma unroll
                        for (int i = 0; i < 2 * kUnits; ++i, src += qstep) cp_async16(d + i * (16 / kUnits) * GB, src);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < kUnits; ++i, src += qstep) cp_async16(d + i * (32 / kUnits) * GB, src);
                }
            } else {
                const uint32_t dst = ring + pat;
                int r = r0, c = c0;
#pragma unroll 1
                for (int i = 0; i < units; i += 3)
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const int u = c >= kUnits;
                        if (pg + u < mine)
                            cp_async16(dst + (uint32_t)(u * (kRows * GB) + r * GB + (c - u * kUnits) * 16), src + (ptrdiff_t)(min(r, last) - r0) * row_bytes + (c - c0) * 16);
                        r += rstep;
                        c += 2;                                               // 32 = 10 * 3 + 2 = 5 * 6 + 2
                        if (c >= units) {
                            c -= units;
                            ++r;
                        }
                    }
            }
            pat += stage_bytes;
            if (pat == ring_bytes) pat = 0;
            qsrc += sg * GB;
            pg += sg;
            if (pg >= mine) {
                pg = 0;
                ptile += wr_n;
                qsrc += qnext;
            }
        }
    };
    // ---- scales and zero points of the slice, and rows of B of the granules this CTA finishes ----
    // A row of the table holds the slice's groups of one weight row in 4-byte words (an odd number of them: rows lie in different
    // banks), and the group before the first where that is an odd one.  Neighbouring lanes take neighbouring words of a row, and
    // 32 / words rows go with an instruction: what these copies cost is the instructions, and the lines that one touches.
    const int sh = g0 & 1, spitch = p.sc_pitch;                               // bytes
    const uint32_t zoff = (uint32_t)(kRows * spitch);
    uint8_t *sc = smem + p.off_sc;
    const int bpitch = rank * 2 + 16;
    const uint8_t *brows = smem + p.off_b;
#pragma unroll 1
    for (int i = 0; i < stages; ++i) {
        issue();
        if (i == 0) {
            {
                const int words = p.sc_words, rows = words < 32 ? 32 / words : 1, lr = words < 32 ? lane / words : 0, w0 = lane - lr * words, wstep = min(words, 32);
                const ptrdiff_t zero = p.zeros - p.scales;
                const __half *scales = p.scales + (g0 - sh);
                if (lr < rows)
#pragma unroll 1
                    for (int r = warp * rows + lr; r < ntiles * kRows; r += kW * rows) {
                        const __half *src = scales + (size_t)min(nrow0 + r, N - 1) * p.G;
                        uint8_t *dst = sc + ((r & ~31) + r) * spitch;
                        if (p.sc_wide)
#pragma unroll 1
                            for (int w = w0; w < words; w += wstep) {
                                if (2 * w >= Gs + sh) break;
                                cp_async4(smem_u32(dst) + 4 * w, src + 2 * w);
                                cp_async4(smem_u32(dst) + zoff + 4 * w, src + zero + 2 * w);
                            }
                        else
#pragma unroll 1
                            for (int i = sh + w0; i < Gs + sh; i += wstep) {
                                *reinterpret_cast<__half *>(dst + 2 * i) = src[i];
                                *reinterpret_cast<__half *>(dst + zoff + 2 * i) = src[zero + i];
                            }
                    }
            }
            if (rank > 0) {
                const int slots = owned(2 * ntiles, cs_log2, crank), c = lane & 15;   // 16-byte unit of a row
#pragma unroll 1
                for (int r = 2 * warp + (lane >> 4); r < 16 * slots; r += 2 * kW) {
                    const int row = min(nrow0 + (((r >> 4) << cs_log2) + crank) * 16 + (r & 15), N - 1);
                    if (c * 8 < rank) cp_async16(smem_u32(brows) + (uint32_t)(r * bpitch + c * 16), static_cast<const T *>(p.B) + (size_t)row * rank + c * 8);
                }
            }
        }
        cp_async_commit();
    }
    uint8_t *xs = smem + kOffX + (size_t)gb * MT * 2048;
    float4 *px = reinterpret_cast<float4 *>(smem + p.off_px) + gb * 4 * MT;
    const T *x = static_cast<const T *>(p.x) + (size_t)(g0 + gb) * kGroupFast;
    T *y = static_cast<T *>(p.y);
    const unsigned long long *twords = p.t;
    const bool wide = p.x_wide != 0;
    const uint8_t *codes0 = smem + p.off_ring + warp * stages * stage_bytes + g * GB + t * (GB / 4);
    const int rq = rank / 2, trow = rank + 16;                                // pairs of words of a token's t; floats of its row in shared memory
    float *s_t = reinterpret_cast<float *>(smem + p.off_t);
    uint8_t *recv0 = smem + p.off_recv;
    const uint32_t pass_bytes = (uint32_t)(((2 * PT + cs - 1) >> cs_log2 << (cs_log2 + wkl)) * MT * 512);
    if (threadIdx.x == 0) mbar_expect_tx(rbar, (uint32_t)(owned(2 * min(PT, ntiles), cs_log2, crank) << (cs_log2 + wkl)) * MT * 512);
    pdl_wait();
    const uint32_t tag = launch_number(sp.epoch);
    constexpr float kScaled = (float)(1 << kUp<BITS, T>);
    uint32_t *overs = reinterpret_cast<uint32_t *>(smem + kOffOver);
    auto over_of = [&](int b) {                                               // of the tokens 8b ..., in this warp's part of the slice
        uint32_t v = 0u;
#pragma unroll 1
        for (int r = b; r < wr_n; r += MT) v |= overs[wk + (r << wkl)];
        return v;
    };
    float up = kScaled;
    bool again = false;
#pragma unroll 1
    for (;;) {
        const uint32_t over = stage_x<BITS, T, MT>(x, K, M, wide, xs, px, mine, wr, wr_n, lane, up);
        cp_async_wait_stage(stages);                                          // the first stage, and with it the scales and B
        if constexpr (kUp<BITS, T> == 0) {
            __syncthreads();
            break;
        }
        if (lane == 0 && !again) overs[warp] = over;
        if (!__syncthreads_or(!again && over != 0)) break;
        again = true;
        up = over_of(wr % MT) >> ((lane >> 3) + (lane & 4)) & 1u ? 1.f : kScaled;
    }
    cluster_wait();                                                           // the other CTAs of the cluster have started

    // ---- granules of 16 rows that this CTA finishes: t.B^T, partial sums added in order, one rounding, store ----
    uint32_t infinite = 0u;                                                   // 0 times the sums, as bits: NaN where one is not finite
    auto finish = [&](int pass) {
        const int pn = min(PT, ntiles - pass * PT), prow0 = nrow0 + pass * PT * kRows, pslot0 = (2 * pass * PT) >> cs_log2;
        uint8_t *rbase = recv0 + (pass & 1) * pass_bytes;
        bool waited = false;
#pragma unroll 1
        for (int it = warp; ; it += kW) {
            const int s = it / MT, b = it - s * MT, gi = (s << cs_log2) + crank, row0 = prow0 + gi * 16;
            if (gi >= 2 * pn || row0 >= N) break;
            float sum[4] = {};
            if (rank > 0) {
                float sub[4][4] = {};
                const uint8_t *bl = brows + ((pslot0 + s) * 16 + g) * bpitch + t * 8;
                const float *tl = s_t + (8 * b + min(g, M - 1 - 8 * b)) * trow + 4 * t;
#pragma unroll 1
                for (int j = 0; j < rank / 16; ++j) {
                    const uint2 b0 = *reinterpret_cast<const uint2 *>(bl + j * 32), b8 = *reinterpret_cast<const uint2 *>(bl + 8 * bpitch + j * 32);
                    const float2 a0 = pair_to_float<T>(b0.x), a1 = pair_to_float<T>(b0.y), c0 = pair_to_float<T>(b8.x), c1 = pair_to_float<T>(b8.y);
                    const float fa[4] = {a0.x, c0.x, a0.y, c0.y}, fb[4] = {a1.x, c1.x, a1.y, c1.y};
                    const float4 v = *reinterpret_cast<const float4 *>(tl + 16 * j);
                    const float e[4] = {v.x, v.y, v.z, v.w};
                    float hi[4], lo[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        hi[i] = __uint_as_float(__float_as_uint(e[i]) & 0xFFFFE000u);
                        lo[i] = hi[i] == e[i] ? 0.f : e[i] - hi[i];           // (an infinite t has no remainder)
                    }
                    mma_tf32(sub[0], fa, hi[0], hi[1]);
                    mma_tf32(sub[1], fa, lo[0], lo[1]);
                    mma_tf32(sub[2], fb, hi[2], hi[3]);
                    mma_tf32(sub[3], fb, lo[2], lo[3]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) sum[c] = (sub[0][c] + sub[2][c]) + (sub[1][c] + sub[3][c]);
            }
            if (!waited && !mbar_wait(rbar + 8u * (pass & 1), (uint32_t)(pass >> 1) & 1u)) atomicExch(sp.status, (int)FBQ_ERR_TIMEOUT);
            waited = true;
            const float4 *src = reinterpret_cast<const float4 *>(rbase) + ((size_t)s << (cs_log2 + wkl)) * MT * 32 + b * 32 + lane;
            float m4[4] = {};
#pragma unroll 1
            for (int c = 0; c < cs << wkl; c += 4) {                          // (four parts at least)
                float4 o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) o[k] = src[(c + k) * MT * 32];
#pragma unroll
                for (int k = 0; k < 4; ++k) { m4[0] += o[k].x; m4[1] += o[k].y; m4[2] += o[k].z; m4[3] += o[k].w; }
            }
            infinite |= __float_as_uint(((m4[0] + m4[1]) + (m4[2] + m4[3])) * 0.f);
            // rows in order through shared memory (the place of this warp's own sums of the granule), whole 16 bytes per store
            T *ybuf = reinterpret_cast<T *>(rbase + ((((size_t)s << (cs_log2 + wkl)) * MT + b) << 9));
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 4; ++c) ybuf[(2 * t + (c & 1)) * 16 + g + 8 * (c >> 1)] = ActTraits<T>::from_float(fmaf(m4[c], 1.f / kScaled, sum[c]));
            __syncwarp();
            const int m = 8 * b + (lane >> 1), n = row0 + 8 * (lane & 1);
            if (lane < 16 && m < M && n < N) *reinterpret_cast<uint4 *>(y + (size_t)m * N + n) = *reinterpret_cast<const uint4 *>(ybuf + lane * 8);
        }
        // Nobody goes on before all sums have arrived: a CTA that left earlier (rows past N, say) would take its shared memory from
        // under stores that are still on their way.
        if (!waited && !mbar_wait(rbar + 8u * (pass & 1), (uint32_t)(pass >> 1) & 1u)) atomicExch(sp.status, (int)FBQ_ERR_TIMEOUT);
    };

    uint4 tw = make_uint4(0u, 0u, 0u, 0u);                                     // (no launch's number: a lane without an early look)
    int slot = 0, mt = 0;                                                     // mt: tiles this warp is through with
#pragma unroll 1
    for (int pass = 0; pass < npass; ++pass) {
        const int pn = min(PT, ntiles - pass * PT);
        const uint32_t recv = smem_u32(recv0) + (pass & 1) * pass_bytes, bar_r = rbar + 8u * (pass & 1);
        if (pass > 1) {
            // sums of this pass go where those of the pass before the last one were: every CTA of the cluster has finished those
            __syncwarp();
            cluster_wait();
        }
        if (pass > 0 && threadIdx.x == 0) mbar_expect_tx(bar_r, (uint32_t)(owned(2 * pn, cs_log2, crank) << (cs_log2 + wkl)) * MT * 512);
#pragma unroll 1
        for (int ti = wr; ti < pn; ti += wr_n, ++mt) {
            if (npass == 1 && mt == my_tiles - 1 && warp < M && lane < rq) tw = load_t2(twords + warp * rank + 2 * lane);     // an early look at t
            float acc[2][MT][4] = {};
            const uint8_t *scl = sc + ((pass * PT + ti) * 2 * kRows + g) * spitch + (sh + gb) * 2;
#pragma unroll 1
            for (int gr = 0; gr < mine; gr += sg) {
                if (mt + gr > 0) {
                    cp_async_wait_stage(stages);
                    __syncwarp();
                }
                const uint8_t *cs0 = codes0 + slot * stage_bytes;
                const uint8_t *xg = xs + (size_t)gr * MT * 2048 + lane * 16, *pg0 = reinterpret_cast<const uint8_t *>(px + gr * 4 * MT + t);
                multiply_group<BITS, T, MT>(cs0, xg, pg0, scl + 2 * gr, zoff, 8 * spitch, acc);
                if (sg == 2 && gr + 1 < mine) multiply_group<BITS, T, MT>(cs0 + kRows * GB, xg + MT * 2048, pg0 + MT * 64, scl + 2 * gr + 2, zoff, 8 * spitch, acc);
                __syncwarp();
                issue();
                cp_async_commit();
                if (++slot == stages) slot = 0;
            }
            if (again) {                                                      // tokens staged with up = 1: the factor that all sums carry
#pragma unroll
                for (int b = 0; b < MT; ++b) {
                    const uint32_t over = over_of(b) >> t;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[h][b][c] *= (over >> (4 * (c & 1))) & 1u ? kScaled : 1.f;
                }
            }
            send_granule<MT>(recv, bar_r, 2 * ti, cs_log2, crank, wkl, wk, lane, acc[0]);
            send_granule<MT>(recv, bar_r, 2 * ti + 1, cs_log2, crank, wkl, wk, lane, acc[1]);
        }
        if (pass == 0 && rank > 0) {
#pragma unroll 1
            for (int m = warp; m < M; m += kW)
#pragma unroll 1
                for (int q = lane; q < rq; q += 32) {
                    uint4 w = tw;
                    if (m != warp || q != lane || w.y != tag || w.w != tag) {
                        const unsigned long long t0 = global_ns();
#pragma unroll 1
                        for (int looks = 1;; ++looks) {
                            w = load_t2(twords + m * rank + 2 * q);
                            if (w.y == tag && w.w == tag) break;
                            if (sp.poll_limit > 0 ? looks >= sp.poll_limit : ((looks & 31) == 0 && global_ns() - t0 > kWaitNs)) {
                                atomicExch(sp.status, (int)FBQ_ERR_TIMEOUT);
                                break;
                            }
                        }
                    }
                    *reinterpret_cast<uint2 *>(s_t + m * trow + q * 2) = make_uint2(w.x, w.z);
                }
            __syncthreads();
        }
        // the pass before, whose sums have arrived meanwhile, and at the end the last one
#pragma unroll 1
        for (int f = max(pass - 1, 0); f < (pass + 1 < npass ? pass : npass); ++f) finish(f);
        if (pass > 0 && pass + 1 < npass) {
            __syncwarp();
            cluster_arrive();
        }
    }
    return (infinite & 0x7F800000u) != 0;
}

// The outputs of this CTA that are not finite once more, product by product.  With an infinite x the sums of (MAGIC + 2^p q) x and P are
// both infinite and their difference is NaN, where a weight times x is infinite; the largest x of bf16 overflow in P alone.
// (What it costs launches that need none of it: 32 x 7 linears of a 7B model, 8 tokens, bf16, 2121 -> 2175 us, 13B layer, 16 tokens, fp16,
// 101.4 -> 101.7; with this in `finish`, where a sum turns out so, 2198 and 103.8.)
template <int BITS, typename T>
__device__ __noinline__ void redo_rows(const SplitDims &p, const uint8_t *smem, int M, int lc, int crank, int cs_log2)
{
    constexpr int NW = BITS == 4 ? 4 : 3;
    const int nrow0 = lc * p.R * kRows, ngran = 2 * min(p.R, p.tiles - lc * p.R);
    T *y = static_cast<T *>(p.y);
#pragma unroll 1
    for (int e = threadIdx.x; e < 16 * M * owned(ngran, cs_log2, crank); e += kThr) {
        const int slot = e / (16 * M), token = e / 16 % M, row = nrow0 + ((slot << cs_log2) + crank) * 16 + e % 16;
        if (row >= p.N || fabsf(ActTraits<T>::to_float(y[(size_t)token * p.N + row])) <= FLT_MAX) continue;
        const uint32_t *w = reinterpret_cast<const uint32_t *>(p.qw) + (size_t)row * p.G * 4 * NW;
        const unsigned short *x = static_cast<const unsigned short *>(p.x) + (size_t)token * p.K;
        float sum = 0.f, sub = 0.f;
#pragma unroll 1
        for (int run = 0; run < 4 * p.G; ++run, w += NW, x += 32) {
            const size_t at = (size_t)row * p.G + (run >> 2);
            const float s = __half2float(p.scales[at]), z = __half2float(p.zeros[at]);
            uint32_t h[16];
            Unpack16<BITS, T>::run(w, h);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int c0 = pair_first<BITS>(j), c1 = pair_second<BITS>(j);
                const float2 q = pair_to_float<T>(h[j]);
                const float down = 1.f / (float)(1 << Unpack16<BITS, T>::div_log2(c0));
                const unsigned short x0 = __ldcg(x + c0), x1 = __ldcg(x + c1);
                sum = fmaf(s * ((q.x - Unpack16<BITS, T>::kMagic) * down - z), ActTraits<T>::to_float(*reinterpret_cast<const T *>(&x0)), sum);
                sum = fmaf(s * ((q.y - Unpack16<BITS, T>::kMagic) * down - z), ActTraits<T>::to_float(*reinterpret_cast<const T *>(&x1)), sum);
            }
        }
        const T *b = reinterpret_cast<const T *>(smem + p.off_b + (slot * 16 + e % 16) * (p.rank * 2 + 16));
        const float *t = reinterpret_cast<const float *>(smem + p.off_t) + token * (p.rank + 16);
#pragma unroll 1
        for (int j = 0; j < p.rank; ++j) sub = fmaf(t[j], ActTraits<T>::to_float(b[j]), sub);
        y[(size_t)token * p.N + row] = ActTraits<T>::from_float(sum + sub);
    }
}

template <int BITS, typename T, int MT>
__global__ void __launch_bounds__(kThr, 1) split_kernel(const __grid_constant__ SplitParams sp)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    pdl_launch_dependents();
    const int cluster = (int)blockIdx.x >> sp.cs_log2, crank = (int)blockIdx.x & ((1 << sp.cs_log2) - 1);
    const bool is_t = cluster < sp.n_tc;
    int pi = 0;
    for (int k = 1; k < sp.n; ++k)
        if (cluster >= (is_t ? sp.first_tc[k] : sp.first_mc[k])) pi = k;
    // The problem's numbers through shared memory: read where they are used they would be one miss of the constant cache after another.
    SplitDims &p = *reinterpret_cast<SplitDims *>(smem + kOffDims);
    if (threadIdx.x < sizeof(SplitDims) / 16) reinterpret_cast<uint4 *>(&p)[threadIdx.x] = reinterpret_cast<const uint4 *>(&sp.p[pi])[threadIdx.x];
    if (threadIdx.x == kThr - 1) {
        mbar_init(smem_u32(smem) + kOffBar, 1u);
        mbar_init(smem_u32(smem) + kOffBar + 8u, 1u);
        fence_barrier_init();
    }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // (the barriers' initialisation has a fence of its own)
    const int g0 = p.G * crank >> sp.cs_log2, Gs = (p.G * (crank + 1) >> sp.cs_log2) - g0;
    if (is_t) {
        const int lc = cluster - p.first_tc;
        if (threadIdx.x == 0) {
            const int ngran = min(p.ngt, (p.rank - lc * p.ngt * 16 + 15) / 16);
            mbar_expect_tx(smem_u32(smem) + kOffBar, (uint32_t)(owned(ngran, sp.cs_log2, crank) << sp.cs_log2) * kTWK * MT * 512u);
        }
        t_program<T, MT>(sp, p, smem, lc, crank, g0, Gs);
        __syncthreads();
    } else {
        if (__syncthreads_or(main_program<BITS, T, MT>(sp, p, smem, cluster - p.first_mc, crank, g0, Gs)))
            redo_rows<BITS, T>(p, smem, sp.M, cluster - p.first_mc, crank, sp.cs_log2);
    }
    // Every CTA read the launch's number before this; with the last one the count of launches goes up by one.  (The CTAs that are
    // through have 32 bits: grids of wide layers, 4096 -> 8 000 000, say, hold more than 65536 CTAs.)
    if (threadIdx.x == 0) atomicAdd(sp.epoch, blockIdx.x == 0 ? (1ull << 32) - (gridDim.x - 1) : 1ull);
}

// ---- host ----------------------------------------------------------------------------------------------------------
struct Shape {
    SplitParams sp{};
    size_t smem = 0;
    int clusters = 0;
    int launches = 1;                        // (several for one problem under a bound: each has `clusters` but the last)
    bool ok = false;
};

// Clusters of CS CTAs that the GPU holds at a time, one CTA per SM (148 SMs; a cluster stays within one of the processing
// clusters, whose SM numbers are no multiples of four).
int resident_clusters(int cs_log2)
{
    static const int n[5] = {148, 74, 33, 15, 6};
    return n[cs_log2];
}
size_t aligned(size_t n, size_t to) { return (n + to - 1) / to * to; }

// Shared memory of a CTA of the problem with p.R tiles, 2^wk_log2 parts of the slice: false where it does not fit.
bool fill_problem(const LinearArgs &a, SplitDims &p, int cs_log2, int wk_log2, size_t *smem)
{
    const int MT = (a.M + 7) / 8, cs = 1 << cs_log2, Gs = (p.G + cs - 1) / cs, mine = (Gs + (1 << wk_log2) - 1) >> wk_log2, wr_n = kW >> wk_log2;
    const size_t x_end = (size_t)kOffX + (size_t)Gs * MT * 2048;
    p.wk_log2 = wk_log2;
    // Half the shared memory for x: what is left beside more of it is a ring of one stage, each copy waited for (81920 -> 1024 at
    // 8 tokens, rank 0: 81 us with 160 KB of x a CTA, 23 with 80).
    if (Gs * MT > 64) return false;
    // a t CTA: x, sums, ring
    p.off_trecv = (int)x_end;
    p.off_tring = (int)aligned(x_end + (aligned(p.ngt, cs) * kTWK * MT) * 512, 128);
    p.tstages = 0;
    if (a.rank > 0) {
        const long room = (long)kSmemAll - p.off_tring;
        p.tstages = (int)std::min<long>({room / (kW * kStageA), (long)kMostStages, (long)(Gs + kTWK - 1) / kTWK});
        if (p.tstages < 1) return false;
        *smem = std::max(*smem, (size_t)p.off_tring + (size_t)p.tstages * kW * kStageA);
    }
    // a main CTA
    size_t at = x_end;
    p.off_px = (int)at;
    at += (size_t)Gs * MT * 64;
    p.off_sc = (int)at;
    p.sc_wide = p.G % 2 == 0 && ((reinterpret_cast<uintptr_t>(a.scales) | reinterpret_cast<uintptr_t>(a.zeros)) & 3) == 0;
    p.sc_words = p.G % (2 * cs) == 0 ? Gs / 2 : (Gs + 2) / 2;                // (where every slice is an even number of groups none begins within a word)
    p.sc_pitch = 4 * (p.sc_words | 1);
    at = aligned(at + (size_t)p.R * 2 * kRows * p.sc_pitch, 16);
    p.off_b = (int)at;
    if (a.rank > 0) at += (size_t)((2 * p.R + cs - 1) >> cs_log2) * 16 * (a.rank * 2 + 16);
    p.off_t = (int)at;
    if (a.rank > 0) at += (size_t)a.M * (a.rank + 16) * 4;
    p.off_recv = (int)at;
    p.sg = mine >= 2 ? 2 : 1;
    size_t stage = (size_t)kW * p.sg * kGroupBytes;
    auto recv = [&](int pt, int nbuf) { return ((size_t)((2 * pt + cs - 1) >> cs_log2) << (cs_log2 + wk_log2)) * MT * 512 * nbuf; };
    p.PT = p.R;
    size_t rb = recv(p.R, 1);
    if (aligned(at + rb, 128) + 2 * stage > kSmemAll && p.R > wr_n) {
        // several passes, two places for their sums; whole rounds of the warps and of the cluster's CTAs
        const int step = std::max(wr_n, cs / 2);
        for (p.PT = (p.R / 2 + step - 1) / step * step; p.PT > step && aligned(at + recv(p.PT, 2), 128) + 2 * stage > kSmemAll; p.PT -= step) {}
        p.PT = std::max(p.PT, step);
        if (p.PT < p.R) rb = recv(p.PT, 2);
        else p.PT = p.R;
    }
    at = aligned(at + rb, 128);
    p.off_ring = (int)at;
    if (p.sg == 2 && at + 2 * stage > kSmemAll) {                            // stages of one group rather than a single stage
        p.sg = 1;
        stage /= 2;
    }
    if (at + stage > kSmemAll) return false;
    const size_t want = (size_t)((p.R + wr_n - 1) / wr_n) * ((mine + p.sg - 1) / p.sg);
    p.stages = (int)std::min<size_t>({(kSmemAll - at) / stage, (size_t)kMostStages, want});
    *smem = std::max(*smem, at + p.stages * stage);
    return true;
}

// Time of a main cluster with q.R tiles (microseconds), 2^w parts of a slice of Gs groups.
double tiles_time(const SplitDims &q, int M, int Gs, int c, int w)
{
    const int MT = (M + 7) / 8, rounds = (q.R + (kW >> w) - 1) / (kW >> w), mine = (Gs + (1 << w) - 1) >> w;
    const bool whole = q.stages * q.sg >= rounds * mine;
    const double units = std::max(q.R * Gs * (0.05 + 0.035 * (MT - 1)), rounds * mine * (0.42 + 0.03 * (MT - 1)));
    const double stream = q.R * Gs * 2.048 / (whole ? 44.0 : std::min(44.0, kW * q.stages * q.sg * 2.048 / 1.3));
    return units + 0.3 * stream + 0.004 * Gs * M + 0.02 * (1 << (w + c)) + 0.01 * rounds * mine + (q.PT < q.R ? 0.5 : 0.0);
}

// One problem under a bound on the CTAs of a grid, those of t among them.  t may take as few clusters as hold it; tiles that a cluster's
// tables do not hold are left to further launches.  The bound goes before the time; a cluster for t and one for the tiles there have
// to be, of as many CTAs as hold x.
Shape make_bounded_shape(const LinearArgs &a, int max_ctas)
{
    Shape best;
    double best_cost = 1e30;
    int best_excess = 1 << 30;
    const int MT = (a.M + 7) / 8, G = a.K / kGroupFast, tiles = (a.N + kRows - 1) / kRows;
    for (int c = 0; c <= (MT == 1 && !best.ok ? 4 : 3) && (1 << c) <= G; ++c)
        for (int ngt = 1;; ngt *= 2) {
            const int n_tc = (a.rank + 16 * ngt - 1) / (16 * ngt), room = std::max(1, std::min(max_ctas >> c, resident_clusters(c)) - n_tc), Gs = (G + (1 << c) - 1) >> c;
            const int excess = std::max(0, ((n_tc + room) << c) - max_ctas);
            bool fits = false;
            for (int R = (tiles + room - 1) / room; R >= 1 && !fits; R = R > 1 ? (R + 1) / 2 : 0)
                for (int w = 3; w >= (c ? 1 : 2); --w) {
                    SplitDims q{};
                    q.N = a.N; q.K = a.K; q.G = G; q.rank = a.rank; q.tiles = tiles; q.R = R; q.ngt = ngt;
                    size_t smem = 0;
                    if (!fill_problem(a, q, c, w, &smem)) continue;
                    fits = true;
                    const int all = (tiles + R - 1) / R, launches = (all + room - 1) / room;
                    const double t_time = a.rank > 0 ? 0.4 * ((ngt + kTWR - 1) / kTWR) * ((Gs + kTWK - 1) / kTWK) : 0.0;
                    const double cost = launches * (std::max(tiles_time(q, a.M, Gs, c, w), t_time) + 0.3 * c + 4.0);
                    if (excess > best_excess || (excess == best_excess && cost >= best_cost)) continue;
                    best_excess = excess;
                    best_cost = cost;
                    best.sp = SplitParams{};
                    best.sp.n = 1; best.sp.M = a.M; best.sp.cs_log2 = c; best.sp.n_tc = n_tc;
                    q.first_mc = best.sp.first_mc[0] = n_tc;
                    best.sp.p[0] = q;
                    best.smem = smem;
                    best.launches = launches;
                    best.clusters = n_tc + (all + launches - 1) / launches;
                    best.ok = true;
                }
            if (16 * ngt >= a.rank) break;
        }
    return best;
}

// The plan of a launch.  What is weighed (microseconds; measured on 4096, 5120, 11008 and 13824 wide layers, INT4, 4 to 16
// tokens): staging x of the slice; the groups of the CTA (the SM's pipes) or of its fullest warp (latency); the stream of codes,
// which a ring of few stages cannot keep up (about 1.3 us from request to arrival); sums to add; clusters, which cost more the
// larger they are (and one of four or eight CTAs leaves SMs unused).  4096 -> 11008, 16 tokens, clusters of two, 8, 4, 2 parts
// of the slice: 17.0, 15.2, 14.7 us; 11008 -> 4096, clusters of two, 8 parts, or of four, 2 parts: 4 tokens 12.4, 13.3, 8 tokens
// 13.5, 14.3; 4096 -> 4096, 16 tokens, CTAs of a cluster 1, 2, 4, 8: 9.4, 8.2, 8.8, 9.8.
Shape make_shape(const LinearArgs *a, int count)
{
    Shape best;
    double best_cost = 1e30;
    const int M = a[0].M, MT = (M + 7) / 8;
    int g_min = 1 << 30;
    for (int i = 0; i < count; ++i) g_min = std::min(g_min, a[i].K / kGroupFast);
    // (clusters of sixteen: for one set of eight tokens of more than 65536 inputs, which no smaller cluster holds)
    for (int c = 0; c <= (MT == 1 && !best.ok ? 4 : 3) && (1 << c) <= g_min; ++c) {
        Shape s;
        s.sp.n = count;
        s.sp.M = M;
        s.sp.cs_log2 = c;
        int n_tc = 0, n_tcs[kMostProblems];
        for (int i = 0; i < count; ++i) {
            SplitDims &p = s.sp.p[i];
            p.N = a[i].N; p.K = a[i].K; p.G = a[i].K / kGroupFast; p.rank = a[i].rank;
            p.tiles = (p.N + kRows - 1) / kRows;
            p.ngt = c >= 2 ? 2 : 1;
            n_tcs[i] = (p.rank + 16 * p.ngt - 1) / (16 * p.ngt);
            n_tc += n_tcs[i];
        }
        // tiles per cluster: the least load of the fullest CTA that lets all main clusters be resident
        const int main_room = std::max(count, resident_clusters(c) - n_tc);
        auto slice = [&](int i) { return (s.sp.p[i].G + (1 << c) - 1) >> c; };
        auto tiles_for = [&](int i, int load) { return std::max(1, load / slice(i)); };
        auto total = [&](int load) {
            long n = 0;
            for (int i = 0; i < count; ++i) n += (s.sp.p[i].tiles + tiles_for(i, load) - 1) / tiles_for(i, load);
            return n;
        };
        int lo = 1, hi = 1;
        while (total(hi) > main_room && hi < (1 << 28)) hi *= 2;
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (total(mid) <= main_room) hi = mid;
            else lo = mid + 1;
        }
        double cost = 0;
        bool ok = true;
        int clusters = n_tc, tc = 0;
        for (int i = 0; i < count && ok; ++i) {
            SplitDims &p = s.sp.p[i];
            const int Gs = slice(i), most = std::min(tiles_for(i, lo), p.tiles), n0 = (p.tiles + most - 1) / most;
            double t = 1e30;
            SplitDims pick = p;
            size_t used = 0;
            ok = false;
            // (where the tables of that many tiles do not fit, fewer: some clusters then start when others are through)
            for (int R = (p.tiles + n0 - 1) / n0; R >= 1 && !ok; R = R > 1 ? (R + 1) / 2 : 0)
                for (int w = 3; w >= (c ? 1 : 2); --w) {
                    SplitDims q = p;
                    q.R = R;
                    size_t sm = 0;
                    if (!fill_problem(a[i], q, c, w, &sm)) continue;
                    const double ti = ((most + R - 1) / R) * tiles_time(q, M, Gs, c, w);
                    if (ti < t) {
                        t = ti;
                        pick = q;
                        used = sm;
                        ok = true;
                    }
                }
            if (!ok) break;
            p = pick;
            s.smem = std::max(s.smem, used);
            cost = std::max(cost, t + 0.3 * c);
            s.sp.first_tc[i] = p.first_tc = tc;
            tc += n_tcs[i];
            s.sp.first_mc[i] = p.first_mc = clusters;
            clusters += (p.tiles + p.R - 1) / p.R;
        }
        if (!ok || cost >= best_cost) continue;
        s.sp.n_tc = n_tc;
        s.clusters = clusters;
        s.ok = true;
        best_cost = cost;
        best = s;
    }
    return best;
}

// Plans, kept per host thread: they hold sizes, no addresses.
struct PlanKey {
    int v[5 + 3 * kMostProblems];
    bool operator==(const PlanKey &o) const { return memcmp(v, o.v, sizeof v) == 0; }
};
struct PlanHash {
    size_t operator()(const PlanKey &k) const
    {
        uint64_t h = 0x9E3779B97F4A7C15ull;
        for (int x : k.v) {
            h = (h ^ (uint32_t)x) * 0xD6E8FEB86659FD93ull;
            h ^= h >> 32;
        }
        return (size_t)h;
    }
};
const Shape &shape_for(const LinearArgs *a, int count, int max_ctas)          // (one problem where there is a bound)
{
    static thread_local std::unordered_map<PlanKey, Shape, PlanHash> plans;
    PlanKey k{};
    k.v[0] = count; k.v[1] = a[0].M; k.v[2] = a[0].rank; k.v[3] = max_ctas;
    for (int i = 0; i < count; ++i) {
        k.v[5 + 3 * i] = a[i].N;
        k.v[6 + 3 * i] = a[i].K;
        k.v[7 + 3 * i] = ((reinterpret_cast<uintptr_t>(a[i].scales) | reinterpret_cast<uintptr_t>(a[i].zeros)) & 3) == 0;
    }
    const auto it = plans.find(k);
    if (it != plans.end()) return it->second;
    if (plans.size() >= 256) plans.clear();
    return plans.emplace(k, max_ctas > 0 ? make_bounded_shape(a[0], max_ctas) : make_shape(a, count)).first->second;
}

template <int BITS, typename T, int MT> cudaError_t launch_one(const Shape &s, bool pdl, cudaStream_t st)
{
    auto kern = split_kernel<BITS, T, MT>;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemAll);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(s.clusters << s.sp.cs_log2));
    cfg.blockDim = dim3(kThr);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    unsigned na = 0;
    if (pdl) {
        at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = 1u << s.sp.cs_log2;
    at[na].val.clusterDim.y = 1;
    at[na].val.clusterDim.z = 1;
    ++na;
    cfg.attrs = at;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, kern, s.sp);
}

template <int BITS, typename T> cudaError_t launch_mt(const Shape &s, bool pdl, cudaStream_t st)
{
    return s.sp.M <= 8 ? launch_one<BITS, T, 1>(s, pdl, st) : launch_one<BITS, T, 2>(s, pdl, st);
}
size_t t_words(const LinearArgs &a) { return ((size_t)a.M * a.rank + 15) / 16 * 16; }

}  // namespace

bool split_supported(const LinearArgs &a)
{
    if (a.group != kGroupFast || a.K < kGroupFast || a.K % kGroupFast != 0) return false;
    return a.M >= 1 && a.M <= kSplitMaxM && a.N % 8 == 0 && a.N >= 8 && a.rank % 16 == 0 && a.rank <= 128;
}

bool split_plan_exists(const LinearArgs *a, int count, const GemvTuning &tune)
{
    return count >= 1 && count <= kMostProblems && (count == 1 || tune.max_ctas == 0) && shape_for(a, count, tune.max_ctas).ok;
}

bool split_plan(const LinearArgs &a, const GemvTuning &tune, int *ctas, int *cluster)
{
    const Shape &s = shape_for(&a, 1, tune.max_ctas);
    *ctas = s.clusters << s.sp.cs_log2;
    *cluster = 1 << s.sp.cs_log2;
    return s.ok;
}

size_t split_scratch_bytes(const LinearArgs *a, int count)
{
    size_t words = 16;                                               // the launch number's line
    for (int i = 0; i < count; ++i) words += t_words(a[i]);
    return words * sizeof(unsigned long long);
}

cudaError_t launch_split(const LinearArgs *a, int count, Workspace &ws, const GemvTuning &tune, cudaStream_t st, int *launches)
{
    if (!split_plan_exists(a, count, tune)) return cudaErrorInvalidConfiguration;
    Shape s = shape_for(a, count, tune.max_ctas);
    s.sp.poll_limit = tune.poll_limit;
    s.sp.skip_t = tune.test_skip_arrive;
    s.sp.status = ws.counters + kCtrStatus;
    s.sp.epoch = reinterpret_cast<unsigned long long *>(ws.split);
    size_t words = 16;
    for (int i = 0; i < count; ++i) {
        SplitDims &p = s.sp.p[i];
        p.x_wide = (reinterpret_cast<uintptr_t>(a[i].x) & 31) == 0;
        p.x = a[i].x; p.A = a[i].A; p.B = a[i].B; p.qw = reinterpret_cast<const uint8_t *>(a[i].qw); p.scales = a[i].scales; p.zeros = a[i].zeros; p.y = a[i].y;
        p.t = reinterpret_cast<unsigned long long *>(ws.split) + words;
        words += t_words(a[i]);
    }
    const bool pdl = tune.pdl != 0;
    const int main = s.clusters - s.sp.n_tc;                         // clusters of a launch
    for (int l = 0; l < s.launches; ++l) {
        if (l > 0) {                                                 // the tiles behind those of the launches before
            s.sp.p[0].first_mc = s.sp.n_tc - l * main;
            s.clusters = s.sp.n_tc + std::min(main, (s.sp.p[0].tiles + s.sp.p[0].R - 1) / s.sp.p[0].R - l * main);
        }
        const cudaError_t e = a[0].bits == 4 ? (a[0].bf16 ? launch_mt<4, __nv_bfloat16>(s, pdl, st) : launch_mt<4, __half>(s, pdl, st))
                                             : (a[0].bf16 ? launch_mt<3, __nv_bfloat16>(s, pdl, st) : launch_mt<3, __half>(s, pdl, st));
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaSuccess;
}

}  // namespace fbq

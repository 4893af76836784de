// Shared declarations of the CUDA sources of libfbq (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/fbq.h"

namespace fbq {

constexpr int kGroupFast = 128;   // group size of the decode / prefill kernels (Section 5.1)
constexpr int kMaxRank = 256;
constexpr int kDecodeMaxM = 16, kDecodePreferM = 6;

// Activation-type helpers ---------------------------------------------------
template <typename T> struct ActTraits;
template <> struct ActTraits<__half> {
    using T2 = __half2;
    static __device__ __forceinline__ float to_float(__half v) { return __half2float(v); }
    static __device__ __forceinline__ __half from_float(float v) { return __float2half_rn(v); }
};
template <> struct ActTraits<__nv_bfloat16> {
    using T2 = __nv_bfloat162;
    static __device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
    static __device__ __forceinline__ __nv_bfloat16 from_float(float v) { return __float2bfloat16_rn(v); }
};

// Per-stream scratch space (device memory owned by the library).
struct Workspace {
    float *partial = nullptr;     // split-K partial sums  [SK][M][N]
    size_t partial_floats = 0;
    float *t = nullptr;           // down-projection t = x.A^T, [M][rank] fp32 (kept zero between calls)
    float *t_gen = nullptr;       // t of the generic path (no invariant), grows on demand
    float *tslots = nullptr;      // streaming decode kernel: partial sums of t, one encoded word per entry (all zero between calls)
    size_t tslots_floats = 0;
    size_t t_floats = 0, t_gen_floats = 0;
    int *counters = nullptr;      // [0]=t arrivals [1]=retired tiles [2]=status [3]=t ready [4]=parked; [8..] per tile
    int n_counters = 0;
    void *trace = nullptr;        // optional phase timestamps of the decode kernel (tuning aid)
    void *stage_x = nullptr;      // staging for the host-buffer entry point
    void *stage_y = nullptr;
    size_t stage_x_bytes = 0, stage_y_bytes = 0;
    void *w16 = nullptr;          // dequantised weights of the dense prefill kernel (no invariant)
    size_t w16_bytes = 0;
    uint32_t *tags = nullptr;     // its launch number and tags (starts at zero)
    size_t n_tags = 0;
    void *split = nullptr;        // the split kernel's launch number and words of t, which carry it (starts at zero)
    size_t split_bytes = 0;
    int gemv_ctas = 0;            // option of the stream (fbq_set_stream_option); outlives the buffers
    void *rec = nullptr;          // split operands of the Gram matrix and the reconstruction step (no invariant)
    size_t rec_bytes = 0;
};
constexpr int kCtrT = 0, kCtrDone = 1, kCtrStatus = 2;   // the decode kernel defines the rest

struct LinearArgs {
    const void *x;
    const uint32_t *qw;
    const __half *scales;
    const __half *zeros;
    const void *A;
    const void *B;
    void *y;
    int M, N, K, group, bits, rank;
    bool bf16;
};

// Launchers implemented in the kernel files.  Each returns a cudaError_t from
// the launch and adds the number of kernels it launched to *launches.
cudaError_t launch_pack(const uint8_t *codes, uint32_t *qw, int N, int K, int bits, cudaStream_t s);
cudaError_t launch_unpack(const uint32_t *qw, uint8_t *codes, int N, int K, int bits, cudaStream_t s);
cudaError_t launch_dequant(const uint32_t *qw, const __half *sc, const __half *ze, float *W, int N,
                           int K, int group, int bits, cudaStream_t s);
cudaError_t launch_generic(const LinearArgs &a, Workspace &ws, cudaStream_t s, int *launches);
cudaError_t launch_sub_branch_unfused(const void *x, const void *A, const void *B, void *y, int M, int N, int K, int rank, bool bf16,
                                      Workspace &ws, cudaStream_t s, int *launches);
cudaError_t launch_quantize_feedback(const float *W, const void *A, const void *B, uint8_t *codes, __half *scales,
                                     __half *zeros, float *WF, float *Delta, int N, int K, int group, int bits, int rank,
                                     int ab_kind, cudaStream_t s);
size_t reconstruct_workspace_floats(int N, int K, int rank);
// Scratch of the two: about `budget` bytes at most, beyond what one slab of rows and the rank need.
size_t gram_scratch_bytes(int T, int K, size_t budget);
size_t reconstruct_scratch_bytes(int N, int K, int rank, size_t budget);
int run_gram(const float *X, float *H, int T, int K, size_t budget, void *scratch, int *status, bool pdl, cudaStream_t s, int *launches);
int run_reconstruct_step(const float *W, const float *H, float *A, float *B, float lr, float *loss, float *ws, int N, int K,
                         int group, int bits, int rank, size_t budget, void *scratch, int *status, bool pdl, cudaStream_t s,
                         int *launches);

struct DecodeTuning {
    int sk = 0, chunk = 0, depth = 0, max_ctas = 0, pdl = 1;
    int t_ctas = 1;  // 1: t = x.A^T comes from a few CTAs at the head of the grid (M <= 4, one K slice)
    int i8 = 1;      // 1: M <= 2 runs the form whose MMAs take the codes and x as 8-bit integers
};
// Returns cudaErrorInvalidConfiguration when no plan fits (caller falls back).
cudaError_t launch_decode(const LinearArgs &a, Workspace &ws, const DecodeTuning &tune,
                          cudaStream_t s, int *launches);
// Scratch the decode kernel needs for a shape (floats of partial sums, ints of counters).
void decode_workspace_need(const LinearArgs &a, const DecodeTuning &tune, size_t *partial_floats,
                           int *counters);

// The streaming decode kernel (fbq_gemv.cu), one and two tokens.
constexpr int kGemvMaxM = 2;
struct GemvTuning {
    int max_ctas = 0;          // 0: one main CTA per SM
    int pdl = 1;
    int poll_limit = 0;        // 0: default number of looks at the "t complete" counter
    int main_ctas = 0;         // > 0: this many main CTAs (a problem of a batch)
    int test_skip_arrive = 0;  // test switch: the t CTAs do not report their arrival (the wait for t must run out)
};
bool gemv_supported(const LinearArgs &a);
void gemv_workspace_need(const LinearArgs &a, const GemvTuning &tune, size_t *tpart_floats, int *counters);
cudaError_t launch_gemv(const LinearArgs &a, Workspace &ws, const GemvTuning &tune, cudaStream_t s, int *launches);

// Several problems of the streaming kernel in one launch: scratch, then launch.  false where they cannot share one (other
// forms, plans that do not fit): then they are launched one by one.
bool gemv_batch_need(const LinearArgs *a, int count, const GemvTuning &tune, size_t *tslots_floats, int *counters);
cudaError_t launch_gemv_batch(const LinearArgs *a, int count, Workspace &ws, const GemvTuning &tune, cudaStream_t s, int *launches);

// The split kernel (fbq_split.cu): the same domain of widths and ranks, up to kSplitMaxM tokens, one problem or several in
// one launch (cudaErrorInvalidConfiguration: no plan fits).  Scratch: Workspace::split, the status word of the counters.
constexpr int kSplitMaxM = 16;
constexpr int kSplitAnyK = 65536;     // up to eight tokens of this many inputs have a plan, with any N and rank
bool split_supported(const LinearArgs &a);
size_t split_scratch_bytes(const LinearArgs *a, int count);
bool split_plan_exists(const LinearArgs *a, int count, const GemvTuning &tune);
bool split_plan(const LinearArgs &a, const GemvTuning &tune, int *ctas, int *cluster);     // CTAs of the grid, of a cluster
cudaError_t launch_split(const LinearArgs *a, int count, Workspace &ws, const GemvTuning &tune, cudaStream_t s, int *launches);

int decode_batch_max();
bool decode_batch_need(const LinearArgs *a, int count, const int *ctas, const DecodeTuning &tune, size_t *partial_floats,
                       size_t *t_floats, int *counters);
cudaError_t launch_decode_batch(const LinearArgs *a, int count, const int *ctas, Workspace &ws, const DecodeTuning &tune,
                                cudaStream_t s, int *launches);
// The dense prefill kernel (fbq_dense.cu).
struct PrefillTuning {
    int pdl = 1;
    int flag_polls = 0;        // 0: waits for t end by time, else after this many looks
    int test_skip_flag = 0;    // test switch: t is not announced (the wait for it must run out)
};
void dense_workspace_need(const LinearArgs &a, size_t *w16_bytes, size_t *tags, size_t *t_floats);
cudaError_t launch_dense(const LinearArgs &a, Workspace &ws, const PrefillTuning &tune, cudaStream_t s, int *launches);

bool prefill_supported(const LinearArgs &a);
bool prefill_dense(const LinearArgs &a);       // the dense kernel is the faster one for this call (fbq_dense.cu)
void prefill_workspace_need(const LinearArgs &a, int *counters, size_t *t_floats, size_t *partial_floats);
// dense: by the dense kernel, whose scratch (dense_workspace_need) is there
cudaError_t launch_prefill(const LinearArgs &a, bool dense, Workspace &ws, cudaStream_t s, int *launches);

}  // namespace fbq

// Surrogate MLP: sizes, parameter layout and kernel launchers (ko_mlp.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ko_internal.h"

// Launch that may begin while the kernel before it in the stream ends (programmatic
// dependent launch): the network's kernels are 4 to 15 us each and follow each
// other, so a launch's own start-up showed between them.  A kernel launched so
// calls pdl_wait() before it touches memory that kernel wrote, or that it reads.
template <typename... Par, typename... Arg>
cudaError_t launch_after(void (*kernel)(Par...), dim3 grid, int threads, size_t smem, cudaStream_t st, Arg... arg)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Par>(arg)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait()
{
#ifdef __CUDA_ARCH__
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
#endif
}
#endif

constexpr int kSlots = 24;        // position slots
constexpr int kSlotFeat = 7;      // features per slot
constexpr int kGlobals = 8;       // global features
constexpr int kMlpIn = 192;       // 24*7 + 8 = 176, padded to 192
constexpr int kHidden = 256;
constexpr int kMaxK = KO_MAX_KERNELS;

constexpr int kEpiReluBf16 = 0;
constexpr int kEpiF32 = 1;

// Flat FP32 parameter layout: W1 [192 x 256] (k-major), b1 [256], W2 [256 x 256],
// b2, W3 [256 x 256], b3, w4 [256], b4 [1].
constexpr long long kOffW1 = 0;
constexpr long long kOffB1 = kOffW1 + (long long)kMlpIn * kHidden;
constexpr long long kOffW2 = kOffB1 + kHidden;
constexpr long long kOffB2 = kOffW2 + (long long)kHidden * kHidden;
constexpr long long kOffW3 = kOffB2 + kHidden;
constexpr long long kOffB3 = kOffW3 + (long long)kHidden * kHidden;
constexpr long long kOffW4 = kOffB3 + kHidden;
constexpr long long kOffB4 = kOffW4 + kHidden;
constexpr long long kParams = kOffB4 + 1;

cudaError_t ko_mlp_gemm_relu(const uint16_t *A, int lda, const uint16_t *Bt, int ldb, int M, int N, int K,
                             const float *bias, uint16_t *out, int ldo, uint16_t *out_t, int ldt,
                             cudaStream_t st);
// tcgen05 forward layer: out = bf16(relu(A Wt^T + bias)), M % 128 == 0,
// K in {192, 256}, N = 256; *err set to 1 if the MMA completion wait gave up.
cudaError_t ko_mlp_layer_tc(const uint16_t *A, const uint16_t *Wt, int M, int K, const float *bias, uint16_t *out,
                            int *err, cudaStream_t st);
// tcgen05 last hidden layer fused with the output layer: y = a . w4 + b4 with
// a = bf16(relu(A Wt^T + bias)) (not stored), in ko_mlp_out_fwd's summation
// order, so y has the same bits as ko_mlp_layer_tc followed by
// ko_mlp_out_fwd (which is what runs, through `out`, when the fused kernel
// does not fit).  Same shapes as ko_mlp_layer_tc.
cudaError_t ko_mlp_layer_tc_out(const uint16_t *A, const uint16_t *Wt, int M, int K, const float *bias,
                                const uint16_t *w4, const float *b4, uint16_t *out, float *y, int *err,
                                cudaStream_t st);
// tcgen05 training forward layer: also writes out_t = out transposed
// ([256][ldt] BF16, ldt % 8 == 0).  Same shapes as ko_mlp_layer_tc.
cudaError_t ko_mlp_layer_tc_t(const uint16_t *A, const uint16_t *Wt, int M, int K, const float *bias, uint16_t *out,
                              uint16_t *out_t, long long ldt, int *err, cudaStream_t st);
// tcgen05 input gradient with the ReLU's backward pass: g = dz W^T (FP32) where
// act > 0, else 0; out[M][256] = bf16(g) (nullable), out_t[256][ldt] its
// transpose, part[M / 32][256] the column sums of each 32 rows in row order
// (M % 128 == 0, ldt % 8 == 0, K = 256).
cudaError_t ko_mlp_dgrad_tc(const uint16_t *dz, const uint16_t *W, int M, const uint16_t *act, uint16_t *out,
                            uint16_t *out_t, long long ldt, float *part, int *err, cudaStream_t st);
// tcgen05 weight gradient A Bt^T with A [M][Kdim] (row stride lda), Bt [256][Kdim]
// (row stride ldb), M <= 256, Kdim % 256 == 0: split-K, one partial matrix
// [256][256] per 256-wide slice in `work` (ko_mlp_wgrad_tc_floats floats), for
// ko_mlp_finish to add up in slice order.
int ko_mlp_wgrad_tc_slices(long long Kdim);
size_t ko_mlp_wgrad_tc_floats(long long Kdim);
cudaError_t ko_mlp_wgrad_tc(const uint16_t *A, long long lda, const uint16_t *Bt, long long ldb, int M,
                            long long Kdim, float *work, int *err, cudaStream_t st);
cudaError_t ko_mlp_gemm_f32(const uint16_t *A, int lda, const uint16_t *Bt, int ldb, int M, int N, int K,
                            float *out, int ldo, cudaStream_t st);
// Encoded orders (rows of one set) x [B x 192].
cudaError_t ko_mlp_encode(const int8_t *rows, int row_stride, const int *set_n, const float *kfeat,
                          const float *gfeat, int B, uint16_t *x, cudaStream_t st);
// FP32 features x [B x 192] (device, B % 64 == 0) rounded to BF16 (nearest, ties to even) into xb and,
// if xt is non-null, transposed into xt [192 x B].
cudaError_t ko_mlp_features(const float *x, int B, uint16_t *xb, uint16_t *xt, cudaStream_t st);
// A training batch: B uniform picks of the labelled pool (row b takes pool entry
// mix64(seed + b golden) % pool), their encoded orders x [B x 192] and xt
// [192 x B], and their targets (B % 32 == 0).
cudaError_t ko_mlp_batch(const int8_t *rows, int row_stride, const int *sid, const float *targets, long long pool,
                         unsigned long long seed, const int *set_n, const float *kfeat, const float *gfeat, int B,
                         uint16_t *x, uint16_t *xt, float *t, cudaStream_t st);
cudaError_t ko_mlp_out_fwd(const uint16_t *a3, const uint16_t *w4, const float *b4, int B, float *y,
                           cudaStream_t st);
// Partial sums of the backward pass, one row per 32 batch rows: [514] of the
// output layer (dw4, db3, loss, db4), then [256] each of db2 and db1.
constexpr int kPartOut = 2 * kHidden + 2;
inline size_t ko_mlp_part_rows(int B) { return (size_t)(B + 31) / 32; }
// Output layer of a training step: y, and dZ3 (row-major and transposed) with
// its partial sums into part [rows x 514].
cudaError_t ko_mlp_out_train(const uint16_t *a3, const uint16_t *w4, const float *b4, const float *t, int B, float *y,
                             uint16_t *dz, uint16_t *dzt, float *part, cudaStream_t st);
// dZ = dA where a > 0, row-major and transposed, column sums per 32 rows into part.
cudaError_t ko_mlp_relu_bwd(const float *da, const uint16_t *a, int B, uint16_t *dz, uint16_t *dzt, float *part,
                            cudaStream_t st);
// End of a backward pass: gradients into g -- a weight matrix from its `slices`
// split-K partials (null: already in g), biases, w4 and the loss sum from the
// partial rows, everything added in a fixed order -- and, with adam.on, one
// Adam step on p, m, v and the BF16 copies the GEMMs read.
struct KoMlpAdam {
    bool on;
    float *p, *m, *v;
    uint16_t *w1t, *w2, *w2t, *w3, *w3t, *w4b;
    float lr, b1, b2, eps, c1, c2;
};
cudaError_t ko_mlp_finish(float *g, const float *wg1, const float *wg2, const float *wg3, int slices,
                          const float *part_out, const float *part2, const float *part1, int B, float *loss_sum,
                          const KoMlpAdam &adam, cudaStream_t st);
cudaError_t ko_mlp_weights_bf16(const float *w, int K, int N, uint16_t *wk, uint16_t *wt, cudaStream_t st);
cudaError_t ko_mlp_topk(const float *y, long long n, int k, uint32_t *state, unsigned int *hist,
                        unsigned int *counters, int *out, cudaStream_t st);
cudaError_t ko_mlp_random_orders(int8_t *rows, int stride, long long count, int n, unsigned long long seed,
                                 cudaStream_t st);
cudaError_t ko_mlp_targets(const int64_t *ms, const int *sid, const double *log2_lb, long long n, float *t,
                           cudaStream_t st);
cudaError_t ko_mlp_neighbours(const int8_t *base, int beam, int n, int8_t *out, cudaStream_t st);
// One step of a steepest descent on the device: `ms` holds the makespans of the
// `nq` neighbours of s->order in `rows` (those ko_mlp_neighbours would write,
// stride 24) and, in its first step, of the order itself behind them.  Moves to
// the best strictly better neighbour (the lowest index among equal ones) and
// writes its neighbours, or ends the descent; rows of an ended one are no orders
// (-1), which an evaluation passes over.
struct KoDescent {
    int64_t makespan;     // of `order`; < 0 before the first step
    int64_t evals;
    int32_t steps, max_steps;
    int32_t done, failed;
    int8_t order[kMaxK];
};
cudaError_t ko_mlp_descend(KoDescent *s, const int64_t *ms, int nq, int n, int8_t *rows, cudaStream_t st);
cudaError_t ko_mlp_gather_rows(const int8_t *src, int stride, const int *pick, int B, int8_t *dst,
                               cudaStream_t st);

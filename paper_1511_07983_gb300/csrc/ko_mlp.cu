// Surrogate MLP kernels: BF16 tensor-core GEMMs with FP32 accumulation and
// fused epilogues, plus the small elementwise kernels of training and
// inference.  The network is 192 -> 256 -> 256 -> 256 -> 1 with ReLU; it
// predicts log2(makespan / lower bound) of a launch order from position-
// ordered kernel descriptors (not part of the paper: a proposal generator for
// sets too large to enumerate, whose proposals are rescored exactly).
//
// The GEMMs here are the warp-level mma.sync path; the tcgen05 kernels of
// ko_mlp_tc.cu run every GEMM whose sizes their tiles divide, and these take
// the rest (batches that are not multiples of 128, or 256 for weight
// gradients) and serve as the cross-check in tests.
//
// GEMM form used everywhere ("NT"): C[m][n] = sum_k A[m][k] * B[n][k], both
// operands K-contiguous BF16 in global memory.  Forward layers take
// B = W^T (stored n-major), input gradients take B = W (k-major), weight
// gradients take A = activations^T and B = dZ^T (both stored transposed by
// the producing kernels).  Tiles: 64 x 128 x 32 per block of 4 warps (each
// warp 32 x 64 = 2 x 8 mma.m16n8k16 tiles), three-stage cp.async pipeline,
// ldmatrix fragment loads from padded shared memory.
#include <cuda_bf16.h>

#include "ko_mlp.h"

namespace {

constexpr int BM = 64, BN = 128, BK = 32, STAGES = 3;
constexpr int PAD = 8;                 // bf16 elements of row padding (16 B): conflict-free ldmatrix
constexpr int LDS = BK + PAD;          // shared-memory row length in elements

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3,
                                            const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(smem_u32(p)));
}

__device__ __forceinline__ void mma_bf16(float *d, const uint32_t *a, const uint32_t *b)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// round-to-nearest-even float -> bf16 bits (explicit bit arithmetic)
__device__ __forceinline__ uint16_t bf16_bits(float x)
{
    uint32_t u = __float_as_uint(x);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}
__device__ __forceinline__ float bf16_val(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

struct Epi {
    int mode;                  // kEpiReluBf16 or kEpiF32
    const float *bias;         // [N] (relu mode)
    uint16_t *out_bf16;        // [M x ldo]
    uint16_t *out_bf16_t;      // [N x ldt] transposed copy, nullable
    float *out_f32;            // [M x ldo] (f32 mode)
    int ldo, ldt;
};

__global__ void __launch_bounds__(128)
gemm_nt_kernel(const uint16_t *__restrict__ A, int lda, const uint16_t *__restrict__ B, int ldb, int M,
               int N, int K, Epi ep)
{
    __shared__ __align__(16) uint16_t sA[STAGES][BM][LDS];
    __shared__ __align__(16) uint16_t sB[STAGES][BN][LDS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 1, wn = warp & 1;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int ktiles = K / BK;

    auto load_stage = [&](int stage, int kt) {
        const int k0 = kt * BK;
#pragma unroll
        for (int i = 0; i < 2; i++) {  // A: 64 rows x 4 chunks of 8 bf16
            const int c = tid + i * 128, row = c >> 2, ch = c & 3;
            cp_async16(&sA[stage][row][ch * 8], A + (size_t)(m0 + row) * lda + k0 + ch * 8);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {  // B: 128 rows x 4 chunks
            const int c = tid + i * 128, row = c >> 2, ch = c & 3;
            cp_async16(&sB[stage][row][ch * 8], B + (size_t)(n0 + row) * ldb + k0 + ch * 8);
        }
    };

    float acc[2][8][4];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 8; j++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[i][j][q] = 0.0f;

#pragma unroll
    for (int s = 0; s < STAGES - 1; s++) {
        if (s < ktiles) load_stage(s, s);
        cp_async_commit();
    }
    for (int kt = 0; kt < ktiles; kt++) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();
        const int nk = kt + STAGES - 1;
        if (nk < ktiles) load_stage(nk % STAGES, nk);
        cp_async_commit();
        const int st = kt % STAGES;
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            uint32_t af[2][4], bfr[8][2];
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const int row = wm * 32 + i * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
                const int col = kk + (lane >> 4) * 8;
                ldmatrix_x4(af[i][0], af[i][1], af[i][2], af[i][3], &sA[st][row][col]);
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int row = wn * 64 + j * 16 + (lane & 7) + (lane >> 4) * 8;
                const int col = kk + ((lane >> 3) & 1) * 8;
                ldmatrix_x4(bfr[2 * j][0], bfr[2 * j][1], bfr[2 * j + 1][0], bfr[2 * j + 1][1],
                            &sB[st][row][col]);
            }
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 8; j++) mma_bf16(acc[i][j], af[i], bfr[j]);
        }
    }
    cp_async_wait<0>();

    // epilogue
#pragma unroll
    for (int i = 0; i < 2; i++) {
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int col = n0 + wn * 64 + j * 8 + (lane & 3) * 2;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int row = m0 + wm * 32 + i * 16 + (lane >> 2) + h * 8;
                float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
                if (ep.mode == kEpiReluBf16) {
                    v0 = fmaxf(v0 + ep.bias[col], 0.0f);
                    v1 = fmaxf(v1 + ep.bias[col + 1], 0.0f);
                    const uint16_t b0 = bf16_bits(v0), b1 = bf16_bits(v1);
                    *(uint32_t *)&ep.out_bf16[(size_t)row * ep.ldo + col] = (uint32_t)b0 | ((uint32_t)b1 << 16);
                    if (ep.out_bf16_t) {
                        ep.out_bf16_t[(size_t)col * ep.ldt + row] = b0;
                        ep.out_bf16_t[(size_t)(col + 1) * ep.ldt + row] = b1;
                    }
                } else {
                    *(float2 *)&ep.out_f32[(size_t)row * ep.ldo + col] = make_float2(v0, v1);
                }
            }
        }
    }
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// ---------------------------------------------------------------- encoding

// x[b] = features of order rows[b] of set sid[b]: kernel at position p goes to
// slot round(23 p / (N-1)); 7 features per slot; 8 global features; zeros
// elsewhere.  Output bf16 row-major [B x 192] and transposed [192 x B].
// Position of an N-kernel order whose slot is `slot`, or -1 (the slots of
// distinct positions are distinct): slot(p) = (2*23*p + (n-1)) / (2(n-1)),
// inverted by testing the positions nearest to slot*(n-1)/23.
__device__ __forceinline__ int slot_position(int n, int slot)
{
    if (n <= 1) return n == 1 && slot == 0 ? 0 : -1;
    const int p0 = (slot * (n - 1)) / (kSlots - 1);
    int pos = -1;
    for (int p = p0 - 1; p <= p0 + 1; p++)
        if (p >= 0 && p < n && (2 * (kSlots - 1) * p + (n - 1)) / (2 * (n - 1)) == slot) pos = p;
    return pos;
}

// Rows of one set.  One thread per row, a warp per 32 consecutive rows.  Per
// block: the slot -> position map of the set's N and its kernel and global
// features.  Per warp step: the 32 rows' order bytes are copied to shared memory
// with coalesced loads;
// each thread produces its row's 192 features in order (slot by slot: one
// kernel index, its 7 features; then the globals and the zero padding),
// packs them two BF16 to a word (round to nearest even) and writes them to a
// per-warp staging area (row pitch 400 bytes: conflict-free 16-byte stores);
// the warp then stores its 32 rows (12,288 contiguous bytes) 16 bytes per
// lane.
constexpr int kEncWarps = 2, kEncPitch = 100;  // staging row pitch in words
__global__ void __launch_bounds__(kEncWarps * 32) encode_kernel(const int8_t *__restrict__ rows, int row_stride,
                                                                const int *__restrict__ set_n,
                                                                const float *__restrict__ kfeat,
                                                                const float *__restrict__ gfeat, int B,
                                                                uint16_t *x)
{
    __shared__ int8_t s_pos[kSlots];
    __shared__ float s_kf[kMaxK * kSlotFeat + kGlobals];
    __shared__ __align__(16) int8_t s_rows[kEncWarps][32 * kMaxK];
    __shared__ __align__(16) uint32_t s_out[kEncWarps][32 * kEncPitch];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();
    for (int i = threadIdx.x; i < kSlots; i += blockDim.x) s_pos[i] = (int8_t)slot_position(set_n[0], i);
    for (int i = threadIdx.x; i < kMaxK * kSlotFeat; i += blockDim.x) s_kf[i] = kfeat[i];
    for (int i = threadIdx.x; i < kGlobals; i += blockDim.x) s_kf[kMaxK * kSlotFeat + i] = gfeat[i];
    __syncthreads();
    const bool stage = row_stride <= kMaxK;
    const long long wsteps = ((long long)B + 31) / 32;
    for (long long ws = (long long)blockIdx.x * kEncWarps + warp; ws < wsteps;
         ws += (long long)gridDim.x * kEncWarps) {
        const int base = (int)(ws * 32), nrows = B - base < 32 ? B - base : 32;
        __syncwarp();  // the previous step's staging has been stored
        if (stage) {
            const int8_t *src = rows + (size_t)base * row_stride;
            const int nb = nrows * row_stride;
            if ((((uintptr_t)src) & 15u) == 0 && (nb & 15) == 0) {
                // 16 bytes per lane: all loads in flight together
                const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
                uint4 *d4 = reinterpret_cast<uint4 *>(s_rows[warp]);
                for (int i = lane; i < nb / 16; i += 32) d4[i] = s4[i];
            } else {
                for (int i = lane; i < nb; i += 32) s_rows[warp][i] = src[i];
            }
            __syncwarp();
        }
        if (lane < nrows) {
            const int8_t *row = stage ? &s_rows[warp][lane * row_stride] : rows + (size_t)(base + lane) * row_stride;
            const float *kf = s_kf, *gf = s_kf + kMaxK * kSlotFeat;
            uint32_t *out = &s_out[warp][lane * kEncPitch];
            float v[8];
            auto put = [&](int f, float val) {  // f is a constant after unrolling
                v[f & 7] = val;
                if ((f & 7) == 7) {
                    uint32_t w[4];
#pragma unroll
                    for (int h = 0; h < 4; h++) {
                        const __nv_bfloat162 p2 = __floats2bfloat162_rn(v[2 * h], v[2 * h + 1]);
                        memcpy(&w[h], &p2, sizeof(uint32_t));
                    }
                    *reinterpret_cast<uint4 *>(out + (f >> 3) * 4) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            };
#pragma unroll
            for (int slot = 0; slot < kSlots; slot++) {
                const int pos = s_pos[slot];
                const int k = pos >= 0 ? (int)row[pos] : -1;
#pragma unroll
                for (int q = 0; q < kSlotFeat; q++) put(slot * kSlotFeat + q, k >= 0 ? kf[k * kSlotFeat + q] : 0.0f);
            }
#pragma unroll
            for (int g = 0; g < kGlobals; g++) put(kSlots * kSlotFeat + g, gf[g]);
#pragma unroll
            for (int f = kSlots * kSlotFeat + kGlobals; f < kMlpIn; f++) put(f, 0.0f);
        }
        __syncwarp();
        // the warp's rows are contiguous in x: 16 bytes per lane per store
        uint4 *dst = reinterpret_cast<uint4 *>(x + (size_t)base * kMlpIn);
        for (int i = lane; i < nrows * (kMlpIn / 8); i += 32) {
            const int r = i / (kMlpIn / 8), c = i % (kMlpIn / 8);
            dst[i] = *reinterpret_cast<const uint4 *>(&s_out[warp][r * kEncPitch + c * 4]);
        }
    }
}

// A training batch.  A block takes 32 rows: 32 threads draw their picks; 768
// (row, slot) pairs look up their kernel; 6,144 features are gathered (the sets'
// tables stay in L1) into a tile whose odd pitch spreads both readings over the
// banks, and leave as 16-byte pieces of rows and as 64-byte runs of the
// transposed copy.  The inference encoder's one thread per row wrote that copy
// two bytes at a time: 18.5 us for 4,096 rows (caches cold) and 5.8 for picks and
// targets in two more kernels; 12.5 us for all of it here.
constexpr int kBatchRows = 32, kBatchPitch = kMlpIn + 2;  // 97 words
__global__ void __launch_bounds__(256) batch_kernel(const int8_t *__restrict__ rows, int row_stride,
                                                    const int *__restrict__ sid, const float *__restrict__ targets,
                                                    long long pool, unsigned long long seed,
                                                    const int *__restrict__ set_n, const float *__restrict__ kfeat,
                                                    const float *__restrict__ gfeat, int B, uint16_t *x, uint16_t *xt,
                                                    float *t)
{
    __shared__ int s_src[kBatchRows], s_set[kBatchRows], s_n[kBatchRows];
    __shared__ int8_t s_kern[kBatchRows][kSlots];
    __shared__ __align__(16) uint16_t tile[kBatchRows * kBatchPitch];
    static_assert(__alignof__(tile) >= sizeof(uint32_t), "read as words below");
    const int r0 = blockIdx.x * kBatchRows;
    pdl_wait();
    if (threadIdx.x < kBatchRows) {
        const int b = r0 + threadIdx.x;
        const int src = (int)(mix64(seed + (unsigned long long)b * 0x9E3779B97F4A7C15ull) % (unsigned long long)pool);
        s_src[threadIdx.x] = src;
        s_set[threadIdx.x] = sid[src];
        s_n[threadIdx.x] = set_n[sid[src]];
        t[b] = targets[src];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBatchRows * kSlots; i += blockDim.x) {
        const int r = i / kSlots, slot = i - r * kSlots;
        const int pos = slot_position(s_n[r], slot);
        s_kern[r][slot] = pos >= 0 ? rows[(size_t)s_src[r] * row_stride + pos] : (int8_t)-1;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBatchRows * kMlpIn; i += blockDim.x) {
        const int r = i / kMlpIn, f = i - r * kMlpIn;
        float v = 0.0f;
        if (f < kSlots * kSlotFeat) {
            const int slot = f / kSlotFeat, k = s_kern[r][slot];
            if (k >= 0) v = kfeat[((size_t)s_set[r] * kMaxK + k) * kSlotFeat + (f - slot * kSlotFeat)];
        } else if (f < kSlots * kSlotFeat + kGlobals) {
            v = gfeat[(size_t)s_set[r] * kGlobals + (f - kSlots * kSlotFeat)];
        }
        tile[r * kBatchPitch + f] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
    __syncthreads();
    const uint32_t *words = reinterpret_cast<const uint32_t *>(tile);
    for (int i = threadIdx.x; i < kBatchRows * (kMlpIn / 8); i += blockDim.x) {
        const int r = i / (kMlpIn / 8), c = i - r * (kMlpIn / 8);
        const uint32_t *w = words + r * (kBatchPitch / 2) + c * 4;
        *reinterpret_cast<uint4 *>(x + (size_t)(r0 + r) * kMlpIn + c * 8) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    for (int i = threadIdx.x; i < kMlpIn * (kBatchRows / 8); i += blockDim.x) {
        const int f = i >> 2, c = (i & 3) * 8;
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; h++)
            w[h] = (uint32_t)tile[(c + 2 * h) * kBatchPitch + f] | ((uint32_t)tile[(c + 2 * h + 1) * kBatchPitch + f] << 16);
        *reinterpret_cast<uint4 *>(xt + (size_t)f * B + r0 + c) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Raw features: FP32 rows [B x 192] to the BF16 operands of the layers -- xb
// row-major, and (training) xt transposed for the weight gradients.  Bound by
// the host link that fills x, not by this pass (B = 65536: 50 MB read, 25 MB
// written).  A block takes 64 rows: coalesced 16-byte reads, 8-byte row stores,
// and the transposed rows leave through shared memory (a 66-element pitch
// spreads a column over the banks) as 128-byte segments.  The host used to
// round and transpose element by element: 24.4 ms of a 65,536-row prediction.
constexpr int kFeatRows = 64, kFeatPitch = kFeatRows + 2;
__global__ void __launch_bounds__(256) features_bf16_kernel(const float *__restrict__ x, int B, uint16_t *xb,
                                                            uint16_t *xt)
{
    __shared__ __align__(16) uint16_t tile[kMlpIn * kFeatPitch];
    static_assert(__alignof__(tile) >= sizeof(uint32_t), "read as words below");
    const long long row0 = (long long)blockIdx.x * kFeatRows;
    constexpr int kQuads = kMlpIn / 4;
    for (int i = threadIdx.x; i < kFeatRows * kQuads; i += blockDim.x) {
        const int r = i / kQuads, f = (i - r * kQuads) * 4;
        const long long at = (row0 + r) * kMlpIn + f;
        const float4 v = __ldcs(reinterpret_cast<const float4 *>(x + at));
        const uint16_t h[4] = {bf16_bits(v.x), bf16_bits(v.y), bf16_bits(v.z), bf16_bits(v.w)};
        *reinterpret_cast<uint2 *>(xb + at) =
            make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16));
        if (xt)
#pragma unroll
            for (int q = 0; q < 4; q++) tile[(f + q) * kFeatPitch + r] = h[q];
    }
    if (!xt) return;
    __syncthreads();
    for (int i = threadIdx.x; i < kMlpIn * (kFeatRows / 2); i += blockDim.x) {
        const int f = i / (kFeatRows / 2), r = (i - f * (kFeatRows / 2)) * 2;
        *reinterpret_cast<uint32_t *>(xt + (long long)f * B + row0 + r) =
            *reinterpret_cast<const uint32_t *>(&tile[f * kFeatPitch + r]);
    }
}

// y[b] = A3[b] . w4 + b4: eight threads per row, thread c sums columns
// 32c .. 32c + 31 as a chain of fused multiply-adds in column order, and the
// eight partials combine as ((p0 + p1) + (p2 + p3)) + ((p4 + p5) + (p6 + p7))
// before b4 is added (the order the fused tcgen05 last layer uses too).
__global__ void out_fwd_kernel(const uint16_t *__restrict__ a3, const uint16_t *__restrict__ w4,
                               const float *__restrict__ b4, int B, float *y)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int b = (int)(i >> 3), c = (int)(i & 7);
    float s = 0.0f;
    if (b < B) {
        const uint4 *src = reinterpret_cast<const uint4 *>(a3 + (size_t)b * kHidden + c * 32);
        const uint16_t *w = w4 + c * 32;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint4 v = src[q];
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int h = 0; h < 4; h++) {
                s = __fmaf_rn(__uint_as_float(u[h] << 16), bf16_val(w[8 * q + 2 * h]), s);
                s = __fmaf_rn(__uint_as_float(u[h] & 0xFFFF0000u), bf16_val(w[8 * q + 2 * h + 1]), s);
            }
        }
    }
    // eight threads of a row sit in one aligned group of eight lanes
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    if (b < B && c == 0) y[b] = s + b4[0];
}

// Output layer of a training step, forward and backward.  y as out_fwd_kernel
// (eight threads per row, its order of sums); dy = 2 (y - t) / B; loss sum;
// dw4 = sum dy * A3; db4 = sum dy; dZ3 = dy * w4 * [A3 > 0] (fp32 for the bias
// gradient, bf16 row-major and transposed for the GEMMs).  A block takes 32
// rows; thread k then walks column k down them, holding the column's sums and
// its 32 BF16 values, which leave as 64 contiguous bytes of the transposed copy
// (two-byte stores before: 30 us for 4,096 rows and 4 for the separate forward
// pass; 6.1 us for both here).  Sums of a block go to part[blockIdx.x]: dw4, db3,
// loss, db4; finish_kernel adds the blocks up in order, so the gradients do not
// depend on the order blocks finish in.
constexpr int kOutRows = 32;
__global__ void __launch_bounds__(kHidden) out_train_kernel(const uint16_t *__restrict__ a3,
                                                            const uint16_t *__restrict__ w4,
                                                            const float *__restrict__ b4, const float *__restrict__ t,
                                                            int B, float *y, uint16_t *dz, uint16_t *dzt, float *part)
{
    __shared__ float s_d[kOutRows], s_dy[kOutRows];
    const int r0 = blockIdx.x * kOutRows, k = threadIdx.x;
    pdl_wait();
    {
        const int r = k >> 3, c = k & 7;
        const uint4 *src = reinterpret_cast<const uint4 *>(a3 + (size_t)(r0 + r) * kHidden + c * 32);
        const uint16_t *w = w4 + c * 32;
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint4 v = src[q];
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int h = 0; h < 4; h++) {
                s = __fmaf_rn(__uint_as_float(u[h] << 16), bf16_val(w[8 * q + 2 * h]), s);
                s = __fmaf_rn(__uint_as_float(u[h] & 0xFFFF0000u), bf16_val(w[8 * q + 2 * h + 1]), s);
            }
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        if (c == 0) {
            const float out = s + b4[0];
            y[r0 + r] = out;
            const float d = out - t[r0 + r];
            s_d[r] = d;
            s_dy[r] = 2.0f * d / (float)B;
        }
    }
    __syncthreads();
    const float w = bf16_val(w4[k]);
    float dw = 0.0f, db = 0.0f;
    uint32_t col[kOutRows / 2];
#pragma unroll
    for (int r = 0; r < kOutRows; r++) {
        const float dy = s_dy[r];
        const float a = bf16_val(a3[(size_t)(r0 + r) * kHidden + k]);
        dw += dy * a;
        const float g = a > 0.0f ? dy * w : 0.0f;
        db += g;
        const uint32_t bits = bf16_bits(g);
        dz[(size_t)(r0 + r) * kHidden + k] = (uint16_t)bits;
        col[r >> 1] = r & 1 ? col[r >> 1] | (bits << 16) : bits;
    }
    uint4 *dt = reinterpret_cast<uint4 *>(dzt + (size_t)k * B + r0);
#pragma unroll
    for (int q = 0; q < 4; q++) dt[q] = make_uint4(col[4 * q], col[4 * q + 1], col[4 * q + 2], col[4 * q + 3]);
    float *mine = part + (size_t)blockIdx.x * kPartOut;
    mine[k] = dw;
    mine[kHidden + k] = db;
    if (k == 0) {
        float lsum = 0.0f, dbsum = 0.0f;
        for (int r = 0; r < kOutRows; r++) {
            lsum += s_d[r] * s_d[r];
            dbsum += s_dy[r];
        }
        mine[2 * kHidden] = lsum;
        mine[2 * kHidden + 1] = dbsum;
    }
}

// Hidden-layer ReLU backward behind the mma.sync input gradient: dZ = dA * [A > 0];
// bias-gradient partials per block (fp32) into part[blockIdx.x]; dZ as bf16
// row-major and transposed.  Thread k walks column k down 32 rows, as above.
__global__ void __launch_bounds__(kHidden) relu_bwd_kernel(const float *__restrict__ da,
                                                           const uint16_t *__restrict__ a, int B, float *part,
                                                           uint16_t *dz, uint16_t *dzt)
{
    const int r0 = blockIdx.x * kOutRows, k = threadIdx.x;
    float db = 0.0f;
    uint32_t col[kOutRows / 2];
#pragma unroll
    for (int r = 0; r < kOutRows; r++) {
        const size_t i = (size_t)(r0 + r) * kHidden + k;
        const float g = bf16_val(a[i]) > 0.0f ? da[i] : 0.0f;
        db += g;
        const uint32_t bits = bf16_bits(g);
        dz[i] = (uint16_t)bits;
        col[r >> 1] = r & 1 ? col[r >> 1] | (bits << 16) : bits;
    }
    uint4 *dt = reinterpret_cast<uint4 *>(dzt + (size_t)k * B + r0);
#pragma unroll
    for (int q = 0; q < 4; q++) dt[q] = make_uint4(col[4 * q], col[4 * q + 1], col[4 * q + 2], col[4 * q + 3]);
    part[(size_t)blockIdx.x * kHidden + k] = db;
}

// Adam on the FP32 master weights.
__device__ __forceinline__ float adam_step(const KoMlpAdam &o, long long i, float gi)
{
    const float mi = o.b1 * o.m[i] + (1.0f - o.b1) * gi;
    const float vi = o.b2 * o.v[i] + (1.0f - o.b2) * gi * gi;
    o.m[i] = mi;
    o.v[i] = vi;
    const float mh = mi / o.c1, vh = vi / o.c2;
    const float pi = o.p[i] - o.lr * mh / (sqrtf(vh) + o.eps);
    o.p[i] = pi;
    return pi;
}

// End of a backward pass (see ko_mlp_finish) in one launch; it took eleven
// (slice sums, partial sums, Adam, BF16 copies; 62 us with cold caches, 14.6 now).  Blocks [0, 176): 32 x 32 tiles
// of the three weight matrices -- a thread adds its elements' slices in order
// (all loads of one element in flight together), updates them and leaves the BF16
// value in a tile from which both layouts are written in 64-byte runs.  The last
// 33 blocks: 32 columns of the per-32-row partials each, loaded by eight warps,
// added in row order by the first.
constexpr int kFinTile = 32, kFinW1 = kMlpIn / kFinTile * (kHidden / kFinTile), kFinW = kHidden / kFinTile * (kHidden / kFinTile);
constexpr int kFinTiles = kFinW1 + 2 * kFinW, kFinSums = (kPartOut + 2 * kHidden + 31) / 32;
constexpr int kFinRows = 128;  // partial rows held at a time
__global__ void __launch_bounds__(256) finish_kernel(float *__restrict__ g, const float *__restrict__ wg1,
                                                     const float *__restrict__ wg2, const float *__restrict__ wg3,
                                                     int slices, const float *__restrict__ part_out,
                                                     const float *__restrict__ part2, const float *__restrict__ part1,
                                                     int nblk, float *loss_sum, const KoMlpAdam o)
{
    __shared__ uint16_t tile[kFinTile][kFinTile + 2];
    __shared__ float rows[kFinRows][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool adam = o.on;
    int blk = blockIdx.x;
    pdl_wait();
    if (blk < kFinTiles) {
        const float *src = wg1;
        long long off = kOffW1;
        uint16_t *wk = nullptr, *wt = o.w1t;
        int K = kMlpIn;
        if (blk >= kFinW1) {
            const bool third = blk >= kFinW1 + kFinW;
            blk -= third ? kFinW1 + kFinW : kFinW1;
            src = third ? wg3 : wg2;
            off = third ? kOffW3 : kOffW2;
            wk = third ? o.w3 : o.w2;
            wt = third ? o.w3t : o.w2t;
            K = kHidden;
        }
        const int k0 = blk / (kHidden / kFinTile) * kFinTile, n0 = blk % (kHidden / kFinTile) * kFinTile;
#pragma unroll
        for (int q = 0; q < kFinTile / 8; q++) {
            const int kr = warp + q * 8;
            const long long i = (long long)(k0 + kr) * kHidden + n0 + lane;
            float gi;
            if (src) {
                gi = 0.0f;
#pragma unroll 8
                for (int s = 0; s < slices; s++) gi += src[(size_t)s * kHidden * kHidden + i];
                g[off + i] = gi;
            } else {
                gi = g[off + i];
            }
            if (adam) {
                const uint16_t b = bf16_bits(adam_step(o, off + i, gi));
                tile[kr][lane] = b;
                if (wk) wk[i] = b;
            }
        }
        if (!adam) return;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kFinTile / 8; q++) {
            const int n = warp + q * 8;
            wt[(size_t)(n0 + n) * K + k0 + lane] = tile[lane][n];
        }
        return;
    }
    // columns: dw4 [0, 256), db3 [256, 512), loss 512, db4 513, db2 [514, 770), db1 [770, 1026)
    const int c = (blk - kFinTiles) * 32 + lane;
    const float *col = nullptr;
    int width = kHidden;
    if (c < kPartOut) { col = part_out + c; width = kPartOut; }
    else if (c < kPartOut + kHidden) col = part2 + (c - kPartOut);
    else if (c < kPartOut + 2 * kHidden) col = part1 + (c - kPartOut - kHidden);
    float acc = 0.0f;
    for (int b0 = 0; b0 < nblk; b0 += kFinRows) {
        const int have = nblk - b0 < kFinRows ? nblk - b0 : kFinRows;
        __syncthreads();
        if (col)
            for (int r = warp; r < have; r += 8) rows[r][lane] = col[(size_t)(b0 + r) * width];
        __syncthreads();
        if (warp == 0 && col)
#pragma unroll 8
            for (int r = 0; r < have; r++) acc += rows[r][lane];
    }
    if (warp != 0 || !col) return;
    if (c == 2 * kHidden) { *loss_sum = acc; return; }
    const long long at = c < kHidden       ? kOffW4 + c
                         : c < 2 * kHidden ? kOffB3 + (c - kHidden)
                         : c < kPartOut    ? kOffB4
                         : c < kPartOut + kHidden ? kOffB2 + (c - kPartOut)
                                                  : kOffB1 + (c - kPartOut - kHidden);
    g[at] = acc;
    if (adam) {
        const float pn = adam_step(o, at, acc);
        if (c < kHidden) o.w4b[c] = bf16_bits(pn);
    }
}

// BF16 copies of one weight matrix W [K x N] (k-major): W itself and W^T.
__global__ void weights_bf16_kernel(const float *__restrict__ w, int K, int N, uint16_t *wk,
                                    uint16_t *wt)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < K * N; i += gridDim.x * blockDim.x) {
        const int k = i / N, n = i % N;
        const uint16_t b = bf16_bits(w[i]);
        if (wk) wk[i] = b;
        if (wt) wt[(size_t)n * K + k] = b;
    }
}

// Order-preserving key of a float (smaller prediction = smaller key).
__device__ __forceinline__ uint32_t float_key(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Radix-select pass: histogram of the next 8-bit digit among keys whose
// higher digits equal the prefix found so far.
__global__ void select_hist_kernel(const float *__restrict__ y, long long n, const uint32_t *state,
                                   int shift, unsigned int *hist)
{
    __shared__ unsigned int h[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const uint32_t prefix = state[0];
    const uint32_t mask = shift == 24 ? 0u : (0xFFFFFFFFu << (shift + 8));
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const uint32_t k = float_key(y[i]);
        if ((k & mask) == (prefix & mask)) atomicAdd(&h[(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// The digit whose bin holds the `need`-th smallest of a 256-bin histogram and how
// many lie below it; one warp, eight bins a lane.
__device__ __forceinline__ void select_digit(const unsigned int *hist, uint32_t need, int &digit, uint32_t &below)
{
    const int lane = threadIdx.x & 31;
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) mine += hist[lane * 8 + i];
    uint32_t upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += v;
    }
    const unsigned has = __ballot_sync(0xffffffffu, upto >= need);
    const int owner = has ? __ffs((int)has) - 1 : 31;
    int d = lane * 8 + 7;
    uint32_t cum = upto - mine;
    for (int i = 0; i < 8; i++) {
        if (cum + hist[lane * 8 + i] >= need) { d = lane * 8 + i; break; }
        if (i < 7) cum += hist[lane * 8 + i];
    }
    digit = __shfl_sync(0xffffffffu, d, owner);
    below = __shfl_sync(0xffffffffu, cum, owner);
}

__global__ void select_init_kernel(uint32_t *state, uint32_t k, unsigned int *hist, unsigned int *counters)
{
    if (threadIdx.x == 0) { state[0] = 0u; state[1] = k; }
    if (threadIdx.x < 2) counters[threadIdx.x] = 0u;
    hist[threadIdx.x] = 0u;
}

// Fix the digit: state = {prefix, remaining k}; clears the histogram.  (One
// thread over 256 bins in memory took 8.7 us of a 13 us digit.)
__global__ void select_scan_kernel(uint32_t *state, int shift, unsigned int *hist)
{
    if (threadIdx.x < 32) {
        int digit;
        uint32_t below;
        const uint32_t need = state[1];
        select_digit(hist, need, digit, below);
        if (threadIdx.x == 0) {
            state[0] |= (uint32_t)digit << shift;
            state[1] = need - below;
        }
    }
    __syncthreads();
    hist[threadIdx.x] = 0;
}

// Up to kSmallTopk keys: the four digits in one block, the keys in shared memory
// (the neighbourhoods of a search round; eight launches, two clears and a copy
// before: 66 of a round's 340 us).
constexpr int kSmallTopk = 8192;
__global__ void __launch_bounds__(1024) select_small_kernel(const float *__restrict__ y, int n, int k, uint32_t *state,
                                                            unsigned int *counters)
{
    __shared__ uint32_t keys[kSmallTopk];
    __shared__ unsigned int hist[256];
    __shared__ uint32_t s_prefix, s_need;
    pdl_wait();
    for (int i = threadIdx.x; i < n; i += blockDim.x) keys[i] = float_key(y[i]);
    if (threadIdx.x == 0) { s_prefix = 0u; s_need = (uint32_t)k; }
    for (int shift = 24; shift >= 0; shift -= 8) {
        if (threadIdx.x < 256) hist[threadIdx.x] = 0u;
        __syncthreads();
        const uint32_t prefix = s_prefix, mask = shift == 24 ? 0u : (0xFFFFFFFFu << (shift + 8));
        for (int i = threadIdx.x; i < n; i += blockDim.x)
            if ((keys[i] & mask) == prefix) atomicAdd(&hist[(keys[i] >> shift) & 255u], 1u);
        __syncthreads();
        if (threadIdx.x < 32) {
            int digit;
            uint32_t below;
            select_digit(hist, s_need, digit, below);
            __syncwarp();
            if (threadIdx.x == 0) {
                s_prefix = prefix | ((uint32_t)digit << shift);
                s_need -= below;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) { state[0] = s_prefix; state[1] = s_need; }
    if (threadIdx.x < 2) counters[threadIdx.x] = 0u;
}

// Write the indices of the k smallest keys: all keys below the threshold and
// `remaining` keys equal to it.
__global__ void select_emit_kernel(const float *__restrict__ y, long long n, const uint32_t *state,
                                   unsigned int *counters, int k, int *out)
{
    const uint32_t thr = state[0], eq_quota = state[1];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const uint32_t key = float_key(y[i]);
        if (key < thr) {
            const unsigned int s = atomicAdd(&counters[0], 1u);
            if (s < (unsigned)k) out[s] = (int)i;
        } else if (key == thr) {
            const unsigned int e = atomicAdd(&counters[1], 1u);
            if (e < eq_quota) {
                const unsigned int s = atomicAdd(&counters[0], 1u);
                if (s < (unsigned)k) out[s] = (int)i;
            }
        }
    }
}

// Uniform random permutations (Fisher-Yates) from a counter-based SplitMix64
// stream per row: row r uses mix64(seed + (r * 2^6 + step) * golden).
__global__ void random_orders_kernel(int8_t *rows, int stride, long long count, int n,
                                     unsigned long long seed)
{
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < count;
         r += (long long)gridDim.x * blockDim.x) {
        int8_t p[kMaxK];
        for (int i = 0; i < n; i++) p[i] = (int8_t)i;
        for (int i = n - 1; i > 0; i--) {
            const unsigned long long x =
                mix64(seed + ((unsigned long long)r * 64ull + (unsigned long long)i) * 0x9E3779B97F4A7C15ull);
            const int j = (int)(x % (unsigned long long)(i + 1));
            const int8_t t = p[i];
            p[i] = p[j];
            p[j] = t;
        }
        for (int i = 0; i < n; i++) rows[r * stride + i] = p[i];
    }
}

// target = log2(makespan / lower bound) as float; invalid makespans give 0.
__global__ void targets_kernel(const int64_t *ms, const int *sid, const double *log2_lb, long long n,
                               float *t)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long m = ms[i];
        t[i] = m > 0 ? (float)(log2((double)m) - log2_lb[sid ? sid[i] : 0]) : 0.0f;
    }
}

// Neighbour q of an n-kernel order: first the n(n-1)/2 swaps of two positions,
// then the n(n-1) moves of one kernel to another position (the rest shift by one).
__device__ __forceinline__ void write_neighbour(const int8_t *base, int n, int q, int8_t *o)
{
    const int swaps = n * (n - 1) / 2;
    int8_t p[kMaxK];
    for (int i = 0; i < n; i++) p[i] = base[i];
    if (q < swaps) {
        int i = 0, rem = q;
        while (rem >= n - 1 - i) { rem -= n - 1 - i; i++; }
        const int j = i + 1 + rem;
        const int8_t t = p[i]; p[i] = p[j]; p[j] = t;
    } else {
        const int m = q - swaps, from = m / (n - 1), k = m % (n - 1);
        const int to = k < from ? k : k + 1;
        const int8_t v = p[from];
        if (from < to) { for (int i = from; i < to; i++) p[i] = p[i + 1]; }
        else { for (int i = from; i > to; i--) p[i] = p[i - 1]; }
        p[to] = v;
    }
    for (int i = 0; i < kMaxK; i++) o[i] = i < n ? p[i] : (int8_t)0;
}

// All single-step neighbours of `beam` base orders (rows of stride 24).  Row r = b * per + q.
__global__ void neighbours_kernel(const int8_t *__restrict__ base, int beam, int n, int8_t *out)
{
    const int per = n * (n - 1) / 2 + n * (n - 1);
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (r >= beam * per) return;
    write_neighbour(base + r / per * kMaxK, n, r % per, out + (size_t)r * kMaxK);
}

// A descent's step between two evaluations.  One block: the step is a few
// microseconds between simulations of hundreds, but the host's part of it (two
// copies back, the choice, two copies and three launches) was 70 of 340.
constexpr int kDescendThreads = 512;
__global__ void __launch_bounds__(kDescendThreads) descend_kernel(KoDescent *s, const int64_t *__restrict__ ms, int nq,
                                                                  int n, int8_t *rows)
{
    __shared__ unsigned long long s_best[kDescendThreads / 32];
    __shared__ int s_idx[kDescendThreads / 32];
    __shared__ int8_t s_order[kMaxK];
    __shared__ int s_done;
    if (s->done) return;
    // the lowest makespan, the lowest index among equal ones; a failed one (< 0) orders below all
    unsigned long long best = ~0ull;
    int at = 0x7fffffff;
    for (int q = threadIdx.x; q < nq; q += kDescendThreads) {
        const unsigned long long v = (unsigned long long)ms[q] ^ (1ull << 63);  // signed order
        if (v < best) { best = v; at = q; }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const unsigned long long b2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int a2 = __shfl_xor_sync(0xffffffffu, at, o);
        if (b2 < best || (b2 == best && a2 < at)) { best = b2; at = a2; }
    }
    if ((threadIdx.x & 31) == 0) { s_best[threadIdx.x >> 5] = best; s_idx[threadIdx.x >> 5] = at; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kDescendThreads / 32; w++)
            if (s_best[w] < best || (s_best[w] == best && s_idx[w] < at)) { best = s_best[w]; at = s_idx[w]; }
        const int64_t found = (int64_t)(best ^ (1ull << 63));
        if (s->makespan < 0) {
            s->makespan = ms[nq];
            s->evals = 1;
        }
        s->evals += nq;
        const bool bad = found < 0 || s->makespan < 0;
        const bool better = !bad && found < s->makespan;
        if (better) {
            s->makespan = found;
            s->steps++;
            for (int i = 0; i < kMaxK; i++) s->order[i] = rows[(size_t)at * kMaxK + i];
        }
        if (bad) s->failed = 1;
        s_done = !better || s->steps >= s->max_steps;
        s->done = s_done;
        for (int i = 0; i < kMaxK; i++) s_order[i] = s->order[i];
    }
    __syncthreads();
    for (int q = threadIdx.x; q <= nq; q += kDescendThreads) {
        if (s_done || q == nq) rows[(size_t)q * kMaxK] = -1;  // row nq: the first order, known now
        else write_neighbour(s_order, n, q, rows + (size_t)q * kMaxK);
    }
}

__global__ void gather_rows_kernel(const int8_t *src, int stride, const int *pick, int B, int8_t *dst)
{
    const int b = blockIdx.x;
    pdl_wait();
    if (b < B && threadIdx.x < stride) dst[(size_t)b * stride + threadIdx.x] = src[(size_t)pick[b] * stride + threadIdx.x];
}

}  // namespace

cudaError_t ko_mlp_gemm_relu(const uint16_t *A, int lda, const uint16_t *Bt, int ldb, int M, int N, int K,
                             const float *bias, uint16_t *out, int ldo, uint16_t *out_t, int ldt,
                             cudaStream_t st)
{
    if (M % BM || N % BN || K % BK) return cudaErrorInvalidValue;
    Epi ep{kEpiReluBf16, bias, out, out_t, nullptr, ldo, ldt};
    gemm_nt_kernel<<<dim3(N / BN, M / BM), 128, 0, st>>>(A, lda, Bt, ldb, M, N, K, ep);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_gemm_f32(const uint16_t *A, int lda, const uint16_t *Bt, int ldb, int M, int N, int K,
                            float *out, int ldo, cudaStream_t st)
{
    if (M % BM || N % BN || K % BK) return cudaErrorInvalidValue;
    Epi ep{kEpiF32, nullptr, nullptr, nullptr, out, ldo, 0};
    gemm_nt_kernel<<<dim3(N / BN, M / BM), 128, 0, st>>>(A, lda, Bt, ldb, M, N, K, ep);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_encode(const int8_t *rows, int row_stride, const int *set_n, const float *kfeat,
                          const float *gfeat, int B, uint16_t *x, cudaStream_t st)
{
    if (B <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long blocks = ((long long)B + 32 * kEncWarps - 1) / (32 * kEncWarps);
    const int grid = (int)(blocks < (long long)sms * 8 ? blocks : (long long)sms * 8);
    ko_count_launch();
    return launch_after(encode_kernel, dim3(grid), kEncWarps * 32, 0, st, rows, row_stride, set_n, kfeat, gfeat, B, x);
}

cudaError_t ko_mlp_batch(const int8_t *rows, int row_stride, const int *sid, const float *targets, long long pool,
                         unsigned long long seed, const int *set_n, const float *kfeat, const float *gfeat, int B,
                         uint16_t *x, uint16_t *xt, float *t, cudaStream_t st)
{
    if (B % kBatchRows) return cudaErrorInvalidValue;
    ko_count_launch();
    return launch_after(batch_kernel, dim3(B / kBatchRows), 256, 0, st, rows, row_stride, sid, targets, pool, seed,
                        set_n, kfeat, gfeat, B, x, xt, t);
}

cudaError_t ko_mlp_features(const float *x, int B, uint16_t *xb, uint16_t *xt, cudaStream_t st)
{
    features_bf16_kernel<<<(unsigned)(B / kFeatRows), 256, 0, st>>>(x, B, xb, xt);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_out_fwd(const uint16_t *a3, const uint16_t *w4, const float *b4, int B, float *y,
                           cudaStream_t st)
{
    out_fwd_kernel<<<(unsigned)(((long long)B * 8 + 255) / 256), 256, 0, st>>>(a3, w4, b4, B, y);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_out_train(const uint16_t *a3, const uint16_t *w4, const float *b4, const float *t, int B, float *y,
                             uint16_t *dz, uint16_t *dzt, float *part, cudaStream_t st)
{
    if (B % kOutRows) return cudaErrorInvalidValue;
    ko_count_launch();
    return launch_after(out_train_kernel, dim3(B / kOutRows), kHidden, 0, st, a3, w4, b4, t, B, y, dz, dzt, part);
}

cudaError_t ko_mlp_relu_bwd(const float *da, const uint16_t *a, int B, uint16_t *dz, uint16_t *dzt, float *part,
                            cudaStream_t st)
{
    if (B % kOutRows) return cudaErrorInvalidValue;
    relu_bwd_kernel<<<(unsigned)(B / kOutRows), kHidden, 0, st>>>(da, a, B, part, dz, dzt);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_finish(float *g, const float *wg1, const float *wg2, const float *wg3, int slices,
                          const float *part_out, const float *part2, const float *part1, int B, float *loss_sum,
                          const KoMlpAdam &adam, cudaStream_t st)
{
    ko_count_launch();
    return launch_after(finish_kernel, dim3(kFinTiles + kFinSums), 256, 0, st, g, wg1, wg2, wg3, slices, part_out,
                        part2, part1, (int)ko_mlp_part_rows(B), loss_sum, adam);
}

cudaError_t ko_mlp_weights_bf16(const float *w, int K, int N, uint16_t *wk, uint16_t *wt, cudaStream_t st)
{
    weights_bf16_kernel<<<256, 256, 0, st>>>(w, K, N, wk, wt);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_topk(const float *y, long long n, int k, uint32_t *state, unsigned int *hist,
                        unsigned int *counters, int *out, cudaStream_t st)
{
    const int blocks = (int)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
    if (n <= kSmallTopk) {
        const cudaError_t e = launch_after(select_small_kernel, dim3(1), 1024, 0, st, y, (int)n, k, state, counters);
        if (e != cudaSuccess) return e;
        ko_count_launch();
    } else {
        select_init_kernel<<<1, 256, 0, st>>>(state, (uint32_t)k, hist, counters);
        ko_count_launch();
        for (int shift = 24; shift >= 0; shift -= 8) {
            select_hist_kernel<<<blocks, 256, 0, st>>>(y, n, state, shift, hist);
            select_scan_kernel<<<1, 256, 0, st>>>(state, shift, hist);
            ko_count_launch(2);
        }
    }
    select_emit_kernel<<<blocks, 256, 0, st>>>(y, n, state, counters, k, out);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_random_orders(int8_t *rows, int stride, long long count, int n, unsigned long long seed,
                                 cudaStream_t st)
{
    long long blocks = (count + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    random_orders_kernel<<<(unsigned)blocks, 256, 0, st>>>(rows, stride, count, n, seed);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_targets(const int64_t *ms, const int *sid, const double *log2_lb, long long n, float *t,
                           cudaStream_t st)
{
    long long blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    targets_kernel<<<(unsigned)blocks, 256, 0, st>>>(ms, sid, log2_lb, n, t);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_neighbours(const int8_t *base, int beam, int n, int8_t *out, cudaStream_t st)
{
    const int per = n * (n - 1) / 2 + n * (n - 1);
    const int rows = beam * per;
    if (rows <= 0) return cudaSuccess;
    ko_count_launch();
    return launch_after(neighbours_kernel, dim3((rows + 127) / 128), 128, 0, st, base, beam, n, out);
}

cudaError_t ko_mlp_descend(KoDescent *s, const int64_t *ms, int nq, int n, int8_t *rows, cudaStream_t st)
{
    descend_kernel<<<1, kDescendThreads, 0, st>>>(s, ms, nq, n, rows);
    ko_count_launch();
    return cudaGetLastError();
}

cudaError_t ko_mlp_gather_rows(const int8_t *src, int stride, const int *pick, int B, int8_t *dst,
                               cudaStream_t st)
{
    ko_count_launch();
    return launch_after(gather_rows_kernel, dim3(B), 32, 0, st, src, stride, pick, B, dst);
}

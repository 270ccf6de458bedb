// Surrogate model: parameters, training on simulator-labelled orders, and
// proposal of orders for sets too large to enumerate, every proposal rescored
// exactly by the run-length simulator.  (The paper has no learned component;
// this serves the same goal as Algorithm 1 -- a good launch order without
// trying all N! -- and every result it returns is an exactly simulated makespan.)
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "ko_fast.h"
#include "ko_mlp.h"

namespace {

constexpr double kBeta1 = 0.9, kBeta2 = 0.999, kEps = 1e-8;

template <typename T>
bool dalloc(T **p, size_t n)
{
    if (cudaMalloc((void **)p, sizeof(T) * (n ? n : 1)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    return true;
}

uint64_t mix64(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// standard normal from two SplitMix64 draws (Box-Muller)
double normal(uint64_t seed, uint64_t i)
{
    const double u1 = ((mix64(seed + (2 * i + 1) * 0x9E3779B97F4A7C15ull) >> 11) + 1.0) * (1.0 / 9007199254740993.0);
    const double u2 = (mix64(seed + (2 * i + 2) * 0x9E3779B97F4A7C15ull) >> 11) * (1.0 / 9007199254740992.0);
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
}

}  // namespace

// Per-set descriptors the encoder reads: kernel features [24][7], globals [8].
void ko_set_features(const KoSet &h, int64_t lb, float *kf, float *gf)
{
    std::memset(kf, 0, sizeof(float) * kMaxK * kSlotFeat);
    for (int i = 0; i < h.n; i++) {
        const KoKern &k = h.k[i];
        float *f = kf + i * kSlotFeat;
        f[0] = (float)((double)k.r / (double)h.R);
        f[1] = (float)((double)k.s / (double)h.Sh);
        f[2] = (float)((double)k.w / (double)h.W);
        f[3] = (float)((double)((k.b + h.S - 1) / h.S) / (double)h.Bk);
        f[4] = (float)(std::log2((double)k.c) / 16.0);
        f[5] = (float)(std::log2((double)k.m) / 16.0);
        f[6] = 1.0f;
    }
    gf[0] = (float)(h.n / 24.0);
    gf[1] = (float)(h.S / 148.0);
    gf[2] = (float)(std::log2((double)h.R) / 24.0);
    gf[3] = (float)(std::log2((double)h.Sh) / 24.0);
    gf[4] = (float)(std::log2((double)h.W) / 24.0);
    gf[5] = (float)(std::log2((double)h.Bk) / 24.0);
    gf[6] = (float)(std::log2((double)(lb > 1 ? lb : 1)) / 32.0);
    gf[7] = 1.0f;
}

struct ko_model {
    float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
    uint16_t *w1t = nullptr, *w2 = nullptr, *w2t = nullptr, *w3 = nullptr, *w3t = nullptr, *w4b = nullptr;
    long long step = 0;
    int cap = 0, cap_wide = 0, cap_train = 0;  // batch capacity of the buffers of a forward pass, of `da`,
                                               // and of the training buffers
    uint16_t *a0 = nullptr, *a0t = nullptr, *a1 = nullptr, *a1t = nullptr, *a2 = nullptr, *a2t = nullptr,
             *a3 = nullptr, *dz = nullptr, *dz2 = nullptr, *dzt = nullptr;
    float *y = nullptr, *t = nullptr, *da = nullptr, *loss = nullptr;
    float *part = nullptr;     // per-32-row partial sums of the backward pass (summed in a fixed order)
    KoFastState fast{};
    int tc_forward = 1;        // inference layers on tcgen05 (1) or mma.sync (0)
    int tc_train = 1;          // training GEMMs on tcgen05 (1) or mma.sync (0)
    float *wg_work = nullptr;  // split-K partials of the tcgen05 weight gradients
    size_t wg_floats = 0;
    int chunk = 262144;        // candidate rows per forward pass of the proposal paths
    int *tc_err = nullptr;     // device flag: a tcgen05 completion wait gave up
    int polish = 64;           // exact descent steps after a guided search (0: none)

    void free_forward()
    {
        cudaFree(a0); cudaFree(a1); cudaFree(a2); cudaFree(a3); cudaFree(y);
        a0 = a1 = a2 = a3 = nullptr;
        y = nullptr;
        cap = 0;
    }
    void free_wide()
    {
        cudaFree(da);
        da = nullptr;
        cap_wide = 0;
    }
    void free_train()
    {
        cudaFree(a0t); cudaFree(a1t); cudaFree(a2t); cudaFree(dz); cudaFree(dz2); cudaFree(dzt); cudaFree(t);
        cudaFree(part);
        a0t = a1t = a2t = dz = dz2 = dzt = nullptr;
        t = part = nullptr;
        cap_train = 0;
    }
    ~ko_model()
    {
        free_forward();
        free_wide();
        free_train();
        cudaFree(p); cudaFree(m); cudaFree(v); cudaFree(g); cudaFree(loss); cudaFree(tc_err); cudaFree(wg_work);
        cudaFree(w1t); cudaFree(w2); cudaFree(w2t); cudaFree(w3); cudaFree(w3t); cudaFree(w4b);
        ko_fast_release(&fast);
    }
};

namespace {

// Activations for a forward pass of B rows.
ko_status ensure_forward(ko_model *md, int B)
{
    if (md->cap >= B) return KO_OK;
    md->free_forward();
    const size_t in = (size_t)B * kMlpIn, hid = (size_t)B * kHidden;
    if (!dalloc(&md->a0, in) || !dalloc(&md->a1, hid) || !dalloc(&md->a2, hid) || !dalloc(&md->a3, hid) ||
        !dalloc(&md->y, (size_t)B)) {
        md->free_forward();
        return KO_ERR_NOMEM;
    }
    md->cap = B;
    return KO_OK;
}

// The FP32 [B x 256] buffer of raw features and mma.sync input gradients.
ko_status ensure_wide(ko_model *md, int B)
{
    if (md->cap_wide >= B) return KO_OK;
    md->free_wide();
    if (!dalloc(&md->da, (size_t)B * kHidden)) return KO_ERR_NOMEM;
    md->cap_wide = B;
    return KO_OK;
}

// Everything a training step of B rows needs.
ko_status ensure_train(ko_model *md, int B)
{
    ko_status s;
    if ((s = ensure_forward(md, B)) || (s = ensure_wide(md, B))) return s;
    if (md->cap_train >= B) return KO_OK;
    md->free_train();
    const size_t in = (size_t)B * kMlpIn, hid = (size_t)B * kHidden;
    if (!dalloc(&md->a0t, in) || !dalloc(&md->a1t, hid) || !dalloc(&md->a2t, hid) || !dalloc(&md->dz, hid) ||
        !dalloc(&md->dz2, hid) || !dalloc(&md->dzt, hid) || !dalloc(&md->t, (size_t)B) ||
        !dalloc(&md->part, ko_mlp_part_rows(B) * (kPartOut + 2 * kHidden))) {
        md->free_train();
        return KO_ERR_NOMEM;
    }
    md->cap_train = B;
    return KO_OK;
}

ko_status cuda_ok(cudaError_t e)
{
    if (e == cudaSuccess) return KO_OK;
    cudaGetLastError();
    return KO_ERR_CUDA;
}

// Two timing events; both null on failure.
static ko_status make_events(cudaEvent_t *e0, cudaEvent_t *e1)
{
    if (cudaEventCreate(e0) != cudaSuccess || cudaEventCreate(e1) != cudaSuccess) {
        cudaGetLastError();
        if (*e0) cudaEventDestroy(*e0);
        *e0 = *e1 = nullptr;
        return KO_ERR_CUDA;
    }
    return KO_OK;
}

ko_status refresh_bf16(ko_model *md, cudaStream_t st)
{
    ko_status s;
    if ((s = cuda_ok(ko_mlp_weights_bf16(md->p + kOffW1, kMlpIn, kHidden, nullptr, md->w1t, st)))) return s;
    if ((s = cuda_ok(ko_mlp_weights_bf16(md->p + kOffW2, kHidden, kHidden, md->w2, md->w2t, st)))) return s;
    if ((s = cuda_ok(ko_mlp_weights_bf16(md->p + kOffW3, kHidden, kHidden, md->w3, md->w3t, st)))) return s;
    return cuda_ok(ko_mlp_weights_bf16(md->p + kOffW4, kHidden, 1, md->w4b, nullptr, st));
}

// Forward over a0 (B rows, B % 64 == 0); with `train` the transposed
// activations for the weight gradients are written too, and the output layer is
// left to backward().
ko_status forward(ko_model *md, int B, bool train, cudaStream_t st)
{
    ko_status s;
    if (train && md->tc_train && B % 128 == 0) {
        // a layer the tcgen05 path cannot take (shared memory) is refused before launch: use mma.sync
        const cudaError_t e = ko_mlp_layer_tc_t(md->a0, md->w1t, B, kMlpIn, md->p + kOffB1, md->a1, md->a1t, B,
                                                md->tc_err, st);
        if (e == cudaSuccess) {
            if ((s = cuda_ok(ko_mlp_layer_tc_t(md->a1, md->w2t, B, kHidden, md->p + kOffB2, md->a2, md->a2t, B,
                                               md->tc_err, st))))
                return s;
            return cuda_ok(ko_mlp_layer_tc(md->a2, md->w3t, B, kHidden, md->p + kOffB3, md->a3, md->tc_err, st));
        }
        if (e != cudaErrorInvalidValue) return cuda_ok(e);
        cudaGetLastError();
        md->tc_train = 0;
    }
    if (!train && md->tc_forward && B % 128 == 0) {
        if ((s = cuda_ok(ko_mlp_layer_tc(md->a0, md->w1t, B, kMlpIn, md->p + kOffB1, md->a1, md->tc_err, st)))) return s;
        if ((s = cuda_ok(ko_mlp_layer_tc(md->a1, md->w2t, B, kHidden, md->p + kOffB2, md->a2, md->tc_err, st)))) return s;
        // the last hidden layer and the output layer in one kernel: a3 is not written
        return cuda_ok(ko_mlp_layer_tc_out(md->a2, md->w3t, B, kHidden, md->p + kOffB3, md->w4b, md->p + kOffB4,
                                           md->a3, md->y, md->tc_err, st));
    }
    if ((s = cuda_ok(ko_mlp_gemm_relu(md->a0, kMlpIn, md->w1t, kMlpIn, B, kHidden, kMlpIn, md->p + kOffB1,
                                      md->a1, kHidden, train ? md->a1t : nullptr, B, st))))
        return s;
    if ((s = cuda_ok(ko_mlp_gemm_relu(md->a1, kHidden, md->w2t, kHidden, B, kHidden, kHidden, md->p + kOffB2,
                                      md->a2, kHidden, train ? md->a2t : nullptr, B, st))))
        return s;
    if ((s = cuda_ok(ko_mlp_gemm_relu(md->a2, kHidden, md->w3t, kHidden, B, kHidden, kHidden, md->p + kOffB3,
                                      md->a3, kHidden, nullptr, 0, st))))
        return s;
    return train ? KO_OK : cuda_ok(ko_mlp_out_fwd(md->a3, md->w4b, md->p + kOffB4, B, md->y, st));
}

// Weight gradient of a layer with activations `at` (transposed, M rows): split-K
// partials on tcgen05 (B % 256 == 0) into *parts, or straight into `out` on mma.sync.
ko_status wgrad(ko_model *md, const uint16_t *at, int M, int B, float *out, float *work, const float **parts,
                cudaStream_t st)
{
    *parts = nullptr;
    if (work) {
        const cudaError_t e = ko_mlp_wgrad_tc(at, B, md->dzt, B, M, B, work, md->tc_err, st);
        if (e == cudaSuccess) *parts = work;
        if (e != cudaErrorInvalidValue) return cuda_ok(e);
        cudaGetLastError();
    }
    return cuda_ok(ko_mlp_gemm_f32(at, B, md->dzt, B, M, kHidden, B, out, kHidden, st));
}

// Gradient of a layer's input times its ReLU's derivative: reads dz, writes dz_out
// (nullable), md->dzt and the bias partials.
ko_status dgrad(ko_model *md, const uint16_t *w, const uint16_t *act, int B, const uint16_t *dz, uint16_t *dz_out,
                float *part, cudaStream_t st)
{
    if (md->tc_train && B % 128 == 0) {
        const cudaError_t e = ko_mlp_dgrad_tc(dz, w, B, act, dz_out, md->dzt, B, part, md->tc_err, st);
        if (e != cudaErrorInvalidValue) return cuda_ok(e);
        cudaGetLastError();
    }
    const ko_status s = cuda_ok(ko_mlp_gemm_f32(dz, kHidden, w, kHidden, B, kHidden, kHidden, md->da, kHidden, st));
    if (s) return s;
    return cuda_ok(ko_mlp_relu_bwd(md->da, act, B, dz_out ? dz_out : md->dz2, md->dzt, part, st));
}

// Output layer, gradients of the mean squared error into md->g and the loss sum
// into *loss_dev; with `adam` an Adam step as well.
ko_status backward(ko_model *md, int B, float *loss_dev, bool adam, float lr, cudaStream_t st)
{
    ko_status s;
    const size_t rows = ko_mlp_part_rows(B);
    float *part_out = md->part, *part2 = part_out + rows * kPartOut, *part1 = part2 + rows * kHidden;
    float *work = nullptr;
    size_t per = 0;
    if (md->tc_train && B % 256 == 0) {
        per = ko_mlp_wgrad_tc_floats(B);
        if (md->wg_floats < 3 * per) {
            cudaFree(md->wg_work);
            md->wg_work = nullptr;
            md->wg_floats = 0;
            if (!dalloc(&md->wg_work, 3 * per)) return KO_ERR_NOMEM;
            md->wg_floats = 3 * per;
        }
        work = md->wg_work;
    }
    const float *wg1, *wg2, *wg3;
    if ((s = cuda_ok(ko_mlp_out_train(md->a3, md->w4b, md->p + kOffB4, md->t, B, md->y, md->dz, md->dzt, part_out, st))))
        return s;
    if ((s = wgrad(md, md->a2t, kHidden, B, md->g + kOffW3, work, &wg3, st))) return s;
    if ((s = dgrad(md, md->w3, md->a2, B, md->dz, md->dz2, part2, st))) return s;
    if ((s = wgrad(md, md->a1t, kHidden, B, md->g + kOffW2, work ? work + per : nullptr, &wg2, st))) return s;
    if ((s = dgrad(md, md->w2, md->a1, B, md->dz2, nullptr, part1, st))) return s;  // no input gradient of layer 1
    if ((s = wgrad(md, md->a0t, kMlpIn, B, md->g + kOffW1, work ? work + 2 * per : nullptr, &wg1, st))) return s;
    KoMlpAdam o{adam,  md->p, md->m, md->v, md->w1t, md->w2, md->w2t, md->w3, md->w3t, md->w4b,
                lr,    (float)kBeta1, (float)kBeta2, (float)kEps, 1.0f, 1.0f};
    if (adam) {
        md->step++;
        o.c1 = (float)(1.0 - std::pow(kBeta1, (double)md->step));
        o.c2 = (float)(1.0 - std::pow(kBeta2, (double)md->step));
    }
    return cuda_ok(ko_mlp_finish(md->g, wg1, wg2, wg3, ko_mlp_wgrad_tc_slices(B), part_out, part2, part1, B, loss_dev,
                                 o, st));
}

// Features of raw rows x [B x 192] (host floats) into a0 and, for training, a0t:
// copied to the device as they are (into `da`, which the backward pass only
// writes later) and rounded there.
ko_status upload_features(ko_model *md, const float *x, int B, bool train, cudaStream_t st)
{
    static_assert(kMlpIn <= kHidden, "the FP32 rows fit the input-gradient buffer");
    if (cudaMemcpyAsync(md->da, x, sizeof(float) * (size_t)B * kMlpIn, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return KO_ERR_CUDA;
    return cuda_ok(ko_mlp_features(md->da, B, md->a0, train ? md->a0t : nullptr, st));
}

}  // namespace

// ---------------------------------------------------------------------- ABI
ko_model *ko_model_new(uint64_t seed, ko_status *err)
{
    ko_model *md = new (std::nothrow) ko_model();
    if (!md) { *err = KO_ERR_NOMEM; return nullptr; }
    bool ok = dalloc(&md->p, kParams) && dalloc(&md->m, kParams) && dalloc(&md->v, kParams) &&
              dalloc(&md->g, kParams) && dalloc(&md->w1t, (size_t)kMlpIn * kHidden) &&
              dalloc(&md->w2, (size_t)kHidden * kHidden) && dalloc(&md->w2t, (size_t)kHidden * kHidden) &&
              dalloc(&md->w3, (size_t)kHidden * kHidden) && dalloc(&md->w3t, (size_t)kHidden * kHidden) &&
              dalloc(&md->w4b, (size_t)kHidden) && dalloc(&md->loss, 1 << 16) && dalloc(&md->tc_err, 1);
    if (!ok) { delete md; *err = KO_ERR_NOMEM; return nullptr; }
    // new device memory holds whatever was there before: the flag must start clear
    if (cudaMemset(md->tc_err, 0, sizeof(int)) != cudaSuccess) { delete md; *err = KO_ERR_CUDA; return nullptr; }
    // He-normal initialisation from a counter-based generator (zero biases,
    // zero weights on the padded input features)
    std::vector<float> h(kParams, 0.0f);
    uint64_t ctr = 0;
    for (int k = 0; k < kMlpIn; k++)
        for (int n = 0; n < kHidden; n++, ctr++)
            h[kOffW1 + (long long)k * kHidden + n] =
                k < kSlots * kSlotFeat + kGlobals ? (float)(normal(seed, ctr) * std::sqrt(2.0 / 176.0)) : 0.0f;
    for (long long i = 0; i < (long long)kHidden * kHidden; i++, ctr++) h[kOffW2 + i] = (float)(normal(seed, ctr) * std::sqrt(2.0 / kHidden));
    for (long long i = 0; i < (long long)kHidden * kHidden; i++, ctr++) h[kOffW3 + i] = (float)(normal(seed, ctr) * std::sqrt(2.0 / kHidden));
    for (int i = 0; i < kHidden; i++, ctr++) h[kOffW4 + i] = (float)(normal(seed, ctr) * std::sqrt(1.0 / kHidden));
    *err = ko_model_load(md, h.data());
    if (*err) { delete md; return nullptr; }
    return md;
}

ko_status ko_model_load(ko_model *md, const float *params)
{
    if (cudaMemcpy(md->p, params, sizeof(float) * kParams, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(md->m, 0, sizeof(float) * kParams) != cudaSuccess ||
        cudaMemset(md->v, 0, sizeof(float) * kParams) != cudaSuccess)
        return KO_ERR_CUDA;
    md->step = 0;
    ko_status s = refresh_bf16(md, nullptr);
    if (s) return s;
    return cudaDeviceSynchronize() == cudaSuccess ? KO_OK : KO_ERR_CUDA;
}

ko_status ko_model_store(const ko_model *md, float *params)
{
    return cudaMemcpy(params, md->p, sizeof(float) * kParams, cudaMemcpyDeviceToHost) == cudaSuccess ? KO_OK
                                                                                                      : KO_ERR_CUDA;
}

void ko_model_free(ko_model *md) { delete md; }

ko_status ko_model_option(ko_model *md, int key, long long value)
{
    if (key == KO_MODEL_OPT_TC) {
        if (value != 0 && value != 1) return KO_ERR_ARG;
        md->tc_forward = (int)value;
        if (cudaMemset(md->tc_err, 0, sizeof(int)) != cudaSuccess) return KO_ERR_CUDA;
        return KO_OK;
    }
    if (key == KO_MODEL_OPT_TC_TRAIN) {
        if (value != 0 && value != 1) return KO_ERR_ARG;
        md->tc_train = (int)value;
        if (cudaMemset(md->tc_err, 0, sizeof(int)) != cudaSuccess) return KO_ERR_CUDA;
        return KO_OK;
    }
    if (key == KO_MODEL_OPT_CHUNK) {
        if (value < 1024 || value > (1 << 22) || value % 1024) return KO_ERR_ARG;
        md->chunk = (int)value;
        return KO_OK;
    }
    if (key == KO_MODEL_OPT_POLISH) {
        if (value < 0 || value > (1 << 20)) return KO_ERR_ARG;
        md->polish = (int)value;
        return KO_OK;
    }
    return KO_ERR_ARG;
}

// KO_ERR_TIMEOUT if a tcgen05 layer reported that its completion wait gave up.
ko_status ko_model_check(ko_model *md)
{
    int e = 0;
    if (cudaMemcpy(&e, md->tc_err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return KO_ERR_CUDA;
    return e ? KO_ERR_TIMEOUT : KO_OK;
}

// Raw features: forward, and optionally backward (+ Adam when lr > 0).
ko_status ko_model_raw(ko_model *md, const float *x, const float *t, int B, float *y_out, float *grad_out,
                       float *loss_out, float lr, cudaStream_t st)
{
    if (B < 64 || B % 64) return KO_ERR_ARG;
    ko_status s = t ? ensure_train(md, B) : ensure_forward(md, B);
    if (!s) s = ensure_wide(md, B);
    if (s) return s;
    if ((s = upload_features(md, x, B, t != nullptr, st))) return s;
    if ((s = forward(md, B, t != nullptr, st))) return s;
    if (t) {
        if (cudaMemcpyAsync(md->t, t, sizeof(float) * B, cudaMemcpyHostToDevice, st) != cudaSuccess)
            return KO_ERR_CUDA;
        if ((s = backward(md, B, md->loss, lr > 0.0f, lr, st))) return s;
        if (grad_out && cudaMemcpyAsync(grad_out, md->g, sizeof(float) * kParams, cudaMemcpyDeviceToHost, st) !=
                            cudaSuccess)
            return KO_ERR_CUDA;
        float ls = 0.0f;
        if (cudaMemcpyAsync(&ls, md->loss, sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return KO_ERR_CUDA;
        if (loss_out) *loss_out = ls / (float)B;
    }
    if (y_out && cudaMemcpyAsync(y_out, md->y, sizeof(float) * B, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return KO_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return KO_ERR_CUDA;
    return ko_model_check(md);
}

// ------------------------------------------------------------ set plumbing

// Parts of one block of memory, 256-byte aligned; without a base it only counts.
struct Carve {
    char *base;
    size_t size = 0;
    explicit Carve(void *b) : base((char *)b) {}
    template <typename T>
    T *take(size_t n)
    {
        const size_t at = size;
        size += (sizeof(T) * (n ? n : 1) + 255) / 256 * 256;
        return base ? (T *)(base + at) : nullptr;
    }
};

// The state's search workspace, at least `bytes` long (nothing of an earlier call
// is in it or in flight on it, see ArenaUse).
static ko_status ensure_arena(KoFastState *fs, size_t bytes)
{
    if (fs->arena_bytes >= bytes) return KO_OK;
    cudaFree(fs->arena);
    fs->arena = nullptr;
    fs->arena_bytes = 0;
    char *p = nullptr;
    if (!dalloc(&p, bytes)) return KO_ERR_NOMEM;
    fs->arena = p;
    fs->arena_bytes = bytes;
    return KO_OK;
}

// End of a call that used the arena: nothing is in flight on it, and no more than
// kArenaKept stays allocated (4M candidates take 120 MB).
constexpr size_t kArenaKept = size_t(256) << 20;
struct ArenaUse {
    KoFastState *fs;
    cudaStream_t st;
    ~ArenaUse()
    {
        cudaStreamSynchronize(st);
        if (fs->arena_bytes <= kArenaKept) return;
        cudaFree(fs->arena);
        fs->arena = nullptr;
        fs->arena_bytes = 0;
    }
};

// Device workspace of a descent over the neighbours of one order.
struct DescentWork {
    KoDescent *state = nullptr;
    int8_t *rows = nullptr;
    int64_t *ms = nullptr;
    KoChunk *chunk = nullptr;
    void carve(Carve &c, int n)
    {
        const size_t per = (size_t)(n * (n - 1) / 2 + n * (n - 1));
        state = c.take<KoDescent>(1);
        rows = c.take<int8_t>((per + 1) * kMaxK);
        ms = c.take<int64_t>(per + 1);
        chunk = c.take<KoChunk>(1);
    }
};
static ko_status descend(KoFastState *fs, const KoSet &h, const int32_t *start, bool moves, int max_iters,
                         int32_t *order_out, int64_t *makespan_out, int32_t *steps_out, int64_t *evals_out,
                         double *gpu_ms, cudaStream_t st, const DescentWork &work);

// Device copies of the sets and what the encoder reads of them, in one block.
struct SetTables {
    void *mem = nullptr;
    int *set_n = nullptr;
    float *kfeat = nullptr, *gfeat = nullptr;
    double *log2_lb = nullptr;
    KoSet *sets = nullptr;
    void carve(Carve &c, int nsets)
    {
        set_n = c.take<int>(nsets);
        kfeat = c.take<float>((size_t)nsets * kMaxK * kSlotFeat);
        gfeat = c.take<float>((size_t)nsets * kGlobals);
        log2_lb = c.take<double>(nsets);
        sets = c.take<KoSet>(nsets);
    }
    ~SetTables() { cudaFree(mem); }
};

static ko_status build_tables(const KoSet *const *hs, int nsets, SetTables *tb, cudaStream_t st)
{
    Carve count(nullptr);
    tb->carve(count, nsets);
    std::vector<char> host(count.size, 0);
    SetTables ht;
    Carve on_host(host.data());
    ht.carve(on_host, nsets);
    for (int i = 0; i < nsets; i++) {
        int64_t lb = 0, ub = 0;
        ko_bounds_host(*hs[i], &lb, &ub);
        ht.set_n[i] = hs[i]->n;
        ko_set_features(*hs[i], lb, ht.kfeat + (size_t)i * kMaxK * kSlotFeat, ht.gfeat + (size_t)i * kGlobals);
        ht.log2_lb[i] = std::log2((double)(lb > 1 ? lb : 1));
        ht.sets[i] = *hs[i];
        ht.sets[i].ref_makespan = 0;
    }
    char *mem = nullptr;
    if (!dalloc(&mem, count.size)) return KO_ERR_NOMEM;
    tb->mem = mem;
    Carve on_device(mem);
    tb->carve(on_device, nsets);
    if (cudaMemcpyAsync(mem, host.data(), host.size(), cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return KO_ERR_CUDA;
    return KO_OK;
}

// Exact makespans of `count` rows (stride 24) of set `set` into out, with the
// choice for that many orders (the state's own options are kept).  `upload`:
// d_chunk does not describe these rows yet.
static ko_status exact_rows(KoFastState *fs, const KoSet *d_sets, const KoSet &h, int set, const int8_t *rows,
                            long long count, int64_t *out, KoChunk *d_chunk, cudaStream_t st, bool upload = true)
{
    KoRoute route(fs, ko_list_choice(h, count), st, true);
    KoChunk c{};
    c.count = count;
    c.set = set;
    c.d0 = h.n;
    c.mode = 2;
    if (upload && cudaMemcpyAsync(d_chunk, &c, sizeof(c), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return KO_ERR_CUDA;
    KoWork w{};
    w.sets = d_sets;
    w.chunks = d_chunk;
    w.nchunks = 1;
    w.n_items = count;
    w.perms = rows;
    w.perm_stride = kMaxK;
    w.out = out;
    w.levels = 1;
    return ko_fast_launch(fs, w, ko_slab_bytes(h.S, h.Bk), st);
}

// Exact makespans of the labelled pool (`per` rows of every set, set after set)
// in one launch per choice: the sets' orders together fill the chip, where 4,096
// orders of one set at a time left most of it idle (32 sets of 6 to 12 kernels:
// a 96-step training run takes 30.9 ms instead of 41.8).
static ko_status label_pool(KoFastState *fs, const KoSet *d_sets, const KoSet *const *hs, int nsets, long long per,
                            const int8_t *rows, int64_t *out, KoChunk *d_chunks, cudaStream_t st)
{
    // the sets by choice, one-thread ones first: each group's chunks follow each other
    std::vector<KoChunk> chunks;
    long long first = 0, lane_items = 0;
    size_t lane_slab = 0, warp_slab = 0;
    int lane_sets = 0;
    for (int lanes : {1, 32}) {
        for (int i = 0; i < nsets; i++) {
            if ((ko_list_choice(*hs[i], per * nsets).lanes == 1) != (lanes == 1)) continue;
            KoChunk c{};
            c.first = first;
            c.count = per;
            c.set = i;
            c.d0 = hs[i]->n;
            c.mode = 2;
            c.list_off = (long long)i * per * kMaxK;
            c.out_off = (long long)i * per;
            chunks.push_back(c);
            first += per;
            size_t &slab = lanes == 1 ? lane_slab : warp_slab;
            slab = std::max(slab, ko_slab_bytes(hs[i]->S, hs[i]->Bk));
        }
        if (lanes == 1) {
            lane_sets = (int)chunks.size();
            lane_items = first;
            first = 0;
        }
    }
    if (cudaMemcpyAsync(d_chunks, chunks.data(), sizeof(KoChunk) * nsets, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return KO_ERR_CUDA;
    for (int lanes : {1, 32}) {
        KoWork w{};
        w.sets = d_sets;
        w.chunks = lanes == 1 ? d_chunks : d_chunks + lane_sets;
        w.nchunks = lanes == 1 ? lane_sets : nsets - lane_sets;
        if (w.nchunks == 0) continue;
        w.n_items = lanes == 1 ? lane_items : first;
        w.perms = rows;
        w.perm_stride = kMaxK;
        w.out = out;
        w.levels = 1;
        KoRoute route(fs, KoChoice{lanes, 1, 0}, st, true);
        const ko_status s = ko_fast_launch(fs, w, lanes == 1 ? lane_slab : warp_slab, st);
        if (s) return s;
    }
    return KO_OK;
}

ko_status ko_model_train_sets(ko_model *md, const KoSet *const *hs, int nsets, long long pairs_per_set,
                              int steps, int batch, float lr, uint64_t seed, float *loss_curve, cudaStream_t st)
{
    if (nsets < 1 || pairs_per_set < 1 || steps < 1 || batch < 64 || batch % 64 || steps > (1 << 16))
        return KO_ERR_ARG;
    for (int i = 0; i < nsets; i++)
        if (!ko_fast_applicable(*hs[i])) return KO_ERR_OVERFLOW;
    SetTables tb;
    ko_status s = build_tables(hs, nsets, &tb, st);
    if (s) return s;
    const long long pool = (long long)nsets * pairs_per_set;
    int8_t *rows = nullptr;
    int64_t *ms = nullptr;
    float *targets = nullptr;
    int *sid = nullptr;
    KoChunk *d_chunks = nullptr;
    if (!dalloc(&rows, (size_t)pool * kMaxK) || !dalloc(&ms, (size_t)pool) || !dalloc(&targets, (size_t)pool) ||
        !dalloc(&sid, (size_t)pool) || !dalloc(&d_chunks, nsets)) {
        cudaFree(rows); cudaFree(ms); cudaFree(targets); cudaFree(sid); cudaFree(d_chunks);
        return KO_ERR_NOMEM;
    }
    std::vector<int> h_sid(pool);
    for (long long i = 0; i < pool; i++) h_sid[i] = (int)(i / pairs_per_set);
    do {
        if (cudaMemcpyAsync(sid, h_sid.data(), sizeof(int) * pool, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaMemsetAsync(rows, 0, (size_t)pool * kMaxK, st) != cudaSuccess) { s = KO_ERR_CUDA; break; }
        // labelled pool: uniform random orders of each set, exact makespans, targets
        for (int i = 0; i < nsets && !s; i++)
            s = cuda_ok(ko_mlp_random_orders(rows + (size_t)i * pairs_per_set * kMaxK, kMaxK, pairs_per_set, hs[i]->n,
                                             mix64(seed ^ (0x5151ull + i)), st));
        if (s) break;
        if ((s = label_pool(&md->fast, tb.sets, hs, nsets, pairs_per_set, rows, ms, d_chunks, st))) break;
        if ((s = cuda_ok(ko_mlp_targets(ms, sid, tb.log2_lb, pool, targets, st)))) break;
        if ((s = ensure_train(md, batch))) break;
        for (int it = 0; it < steps && !s; it++) {
            if ((s = cuda_ok(ko_mlp_batch(rows, kMaxK, sid, targets, pool, mix64(seed + 0x1000ull + it), tb.set_n,
                                          tb.kfeat, tb.gfeat, batch, md->a0, md->a0t, md->t, st))))
                break;
            if ((s = forward(md, batch, true, st))) break;
            s = backward(md, batch, md->loss + it, true, lr, st);
        }
        if (s) break;
        if (loss_curve) {
            std::vector<float> lc(steps);
            if (cudaMemcpyAsync(lc.data(), md->loss, sizeof(float) * steps, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess) { s = KO_ERR_CUDA; break; }
            for (int i = 0; i < steps; i++) loss_curve[i] = lc[i] / (float)batch;
        }
        if (cudaStreamSynchronize(st) != cudaSuccess) s = KO_ERR_CUDA;
        if (!s) s = ko_model_check(md);  // a tcgen05 completion wait that gave up
    } while (false);
    cudaFree(rows); cudaFree(ms); cudaFree(targets); cudaFree(sid); cudaFree(d_chunks);
    return s;
}

// Best exact makespan among the rows [count x 24] of one set (device), index too.
static ko_status best_of(const int64_t *d_ms, long long count, int64_t *best, long long *best_idx)
{
    std::vector<int64_t> h(count);
    if (cudaMemcpy(h.data(), d_ms, sizeof(int64_t) * count, cudaMemcpyDeviceToHost) != cudaSuccess)
        return KO_ERR_CUDA;
    long long bi = -1;
    for (long long i = 0; i < count; i++)
        if (h[i] >= 0 && (bi < 0 || h[i] < h[bi])) bi = i;
    if (bi < 0) return KO_ERR_STATE;
    *best = h[bi];
    *best_idx = bi;
    return KO_OK;
}

// Rows of one forward pass over `rows` candidates: the model's chunk, or all of
// them in whole 128-row tiles where they are fewer.
static int chunk_rows(const ko_model *md, long long rows)
{
    const long long all = (rows + 127) / 128 * 128;
    return all < md->chunk ? (int)all : md->chunk;
}

ko_status ko_model_propose_set(ko_model *md, const KoSet &h, long long n_cand, int top_k, uint64_t seed,
                               int32_t *best_order, int64_t *best_makespan, double *gpu_ms, cudaStream_t st)
{
    if (n_cand < 1 || top_k < 1 || top_k > n_cand || n_cand > (1ll << 26)) return KO_ERR_ARG;
    if (!ko_fast_applicable(h)) return KO_ERR_OVERFLOW;
    const KoSet *hs[1] = {&h};
    SetTables tb;
    ko_status s = build_tables(hs, 1, &tb, st);
    if (s) return s;
    const int C = chunk_rows(md, n_cand);
    const long long padded = (n_cand + C - 1) / C * C;
    int8_t *rows, *top_rows;
    float *y_all;
    int *top_idx;
    int64_t *top_ms;
    uint32_t *sel_state;
    unsigned int *sel_hist, *sel_cnt;
    KoChunk *d_chunk;
    auto carve = [&](Carve &c) {
        rows = c.take<int8_t>((size_t)padded * kMaxK);
        y_all = c.take<float>((size_t)n_cand);
        top_idx = c.take<int>(top_k);
        top_rows = c.take<int8_t>((size_t)top_k * kMaxK);
        top_ms = c.take<int64_t>(top_k);
        sel_state = c.take<uint32_t>(2);
        sel_hist = c.take<unsigned int>(256);
        sel_cnt = c.take<unsigned int>(2);
        d_chunk = c.take<KoChunk>(1);
    };
    Carve need(nullptr);
    carve(need);
    ArenaUse use{&md->fast, st};
    s = ensure_arena(&md->fast, need.size);
    Carve mem(md->fast.arena);
    if (!s) carve(mem);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (!s) s = make_events(&e0, &e1);
    if (!s) s = ensure_forward(md, C);
    if (!s) {
        cudaEventRecord(e0, st);
        if (cudaMemsetAsync(rows, 0, (size_t)padded * kMaxK, st) != cudaSuccess) s = KO_ERR_CUDA;
        if (!s) s = cuda_ok(ko_mlp_random_orders(rows, kMaxK, n_cand, h.n, mix64(seed ^ 0xC0FFEEull), st));
        for (long long off = 0; off < n_cand && !s; off += C) {
            const long long c = n_cand - off < C ? n_cand - off : C;
            if ((s = cuda_ok(ko_mlp_encode(rows + (size_t)off * kMaxK, kMaxK, tb.set_n, tb.kfeat, tb.gfeat, C,
                                           md->a0, st))))
                break;
            if ((s = forward(md, C, false, st))) break;
            if (cudaMemcpyAsync(y_all + off, md->y, sizeof(float) * c, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                s = KO_ERR_CUDA;
        }
        if (!s) s = cuda_ok(ko_mlp_topk(y_all, n_cand, top_k, sel_state, sel_hist, sel_cnt, top_idx, st));
        if (!s) s = cuda_ok(ko_mlp_gather_rows(rows, kMaxK, top_idx, top_k, top_rows, st));
        if (!s) s = exact_rows(&md->fast, tb.sets, h, 0, top_rows, top_k, top_ms, d_chunk, st);
        cudaEventRecord(e1, st);
        if (!s && cudaStreamSynchronize(st) != cudaSuccess) s = KO_ERR_CUDA;
    }
    if (!s) s = ko_model_check(md);
    if (!s) {
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (gpu_ms) *gpu_ms = ms;
        long long bi = 0;
        s = best_of(top_ms, top_k, best_makespan, &bi);
        int8_t r[kMaxK];
        if (!s && cudaMemcpy(r, top_rows + (size_t)bi * kMaxK, kMaxK, cudaMemcpyDeviceToHost) != cudaSuccess)
            s = KO_ERR_CUDA;
        if (!s)
            for (int i = 0; i < h.n; i++) best_order[i] = r[i];
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    return s;
}

// Surrogate-guided local search.  Screening: the network scores n_cand
// uniform random orders, the top_k are rescored exactly, and the `beam` best
// exact orders seed the search.  Each round: every swap and every single move
// of each beam order is scored by the network, the k2 best are rescored
// exactly, and the beam becomes the `beam` best distinct orders seen so far.
// Every reported makespan is exact.
ko_status ko_model_search_set(ko_model *md, const KoSet &h, long long n_cand, int top_k, int rounds, int beam,
                              uint64_t seed, int32_t *best_order, int64_t *best_makespan, double *gpu_ms,
                              cudaStream_t st)
{
    const int n = h.n;
    if (n_cand < 1 || top_k < 1 || top_k > n_cand || n_cand > (1ll << 26) || rounds < 0 || rounds > 1024 ||
        beam < 1 || beam > 64 || n < 2)
        return KO_ERR_ARG;
    if (!ko_fast_applicable(h)) return KO_ERR_OVERFLOW;
    const KoSet *hs[1] = {&h};
    SetTables tb;
    ko_status s = build_tables(hs, 1, &tb, st);
    if (s) return s;
    const int k2 = 256;
    const int per = n * (n - 1) / 2 + n * (n - 1);
    const int nb_rows = beam * per, nb_pad = (nb_rows + 127) / 128 * 128;
    // rows per forward pass: no more than there are (the screening's or a round's)
    const int C = chunk_rows(md, std::max<long long>(n_cand, nb_pad));
    const long long padded = (n_cand + C - 1) / C * C;
    const int kmax = top_k > k2 ? top_k : k2;
    int8_t *rows, *top_rows, *nb, *base;
    float *y_all;
    int *top_idx;
    int64_t *top_ms;
    uint32_t *sel_state;
    unsigned int *sel_hist, *sel_cnt;
    KoChunk *d_chunk;
    DescentWork polish;  // its own: the descent leaves the search's buffers alone
    auto carve = [&](Carve &c) {
        rows = c.take<int8_t>((size_t)padded * kMaxK);
        y_all = c.take<float>((size_t)std::max<long long>(n_cand, nb_pad));
        top_idx = c.take<int>(kmax);
        top_rows = c.take<int8_t>((size_t)kmax * kMaxK);
        top_ms = c.take<int64_t>(kmax);
        nb = c.take<int8_t>((size_t)nb_pad * kMaxK);
        base = c.take<int8_t>((size_t)beam * kMaxK);
        sel_state = c.take<uint32_t>(2);
        sel_hist = c.take<unsigned int>(256);
        sel_cnt = c.take<unsigned int>(2);
        d_chunk = c.take<KoChunk>(1);
        polish.carve(c, n);
    };
    Carve need(nullptr);
    carve(need);
    ArenaUse use{&md->fast, st};
    s = ensure_arena(&md->fast, need.size);
    Carve mem(md->fast.arena);
    if (!s) carve(mem);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    struct Cand {
        int64_t ms;
        std::vector<int8_t> row;
    };
    std::vector<Cand> pool;
    // exact makespans of `cnt` device rows -> pool
    auto collect = [&](int cnt) -> ko_status {
        std::vector<int64_t> hm(cnt);
        std::vector<int8_t> hr((size_t)cnt * kMaxK);
        if (cudaMemcpyAsync(hm.data(), top_ms, sizeof(int64_t) * cnt, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaMemcpyAsync(hr.data(), top_rows, hr.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return KO_ERR_CUDA;
        for (int i = 0; i < cnt; i++)
            if (hm[i] >= 0) pool.push_back(Cand{hm[i], std::vector<int8_t>(hr.begin() + (size_t)i * kMaxK, hr.begin() + (size_t)(i + 1) * kMaxK)});
        std::stable_sort(pool.begin(), pool.end(), [](const Cand &a, const Cand &b) { return a.ms < b.ms; });
        std::vector<Cand> kept;
        for (const Cand &c : pool) {
            bool dup = false;
            for (const Cand &k : kept) dup = dup || k.row == c.row;
            if (!dup) kept.push_back(c);
            if ((int)kept.size() == beam) break;
        }
        pool.swap(kept);
        return KO_OK;
    };
    if (!s) s = make_events(&e0, &e1);
    if (!s) s = ensure_forward(md, C);
    if (!s) {
        cudaEventRecord(e0, st);
        // screening
        if (cudaMemsetAsync(rows, 0, (size_t)padded * kMaxK, st) != cudaSuccess ||
            cudaMemsetAsync(nb, 0, (size_t)nb_pad * kMaxK, st) != cudaSuccess)
            s = KO_ERR_CUDA;
        if (!s) s = cuda_ok(ko_mlp_random_orders(rows, kMaxK, n_cand, n, mix64(seed ^ 0xC0FFEEull), st));
        for (long long off = 0; off < n_cand && !s; off += C) {
            const long long c = n_cand - off < C ? n_cand - off : C;
            if ((s = cuda_ok(ko_mlp_encode(rows + (size_t)off * kMaxK, kMaxK, tb.set_n, tb.kfeat, tb.gfeat, C,
                                           md->a0, st))))
                break;
            if ((s = forward(md, C, false, st))) break;
            if (cudaMemcpyAsync(y_all + off, md->y, sizeof(float) * c, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                s = KO_ERR_CUDA;
        }
        if (!s) s = cuda_ok(ko_mlp_topk(y_all, n_cand, top_k, sel_state, sel_hist, sel_cnt, top_idx, st));
        if (!s) s = cuda_ok(ko_mlp_gather_rows(rows, kMaxK, top_idx, top_k, top_rows, st));
        if (!s) s = exact_rows(&md->fast, tb.sets, h, 0, top_rows, top_k, top_ms, d_chunk, st);
        if (!s) s = collect(top_k);
        // local search rounds
        for (int r = 0; r < rounds && !s && !pool.empty(); r++) {
            const int nbase = (int)pool.size();
            std::vector<int8_t> hb((size_t)nbase * kMaxK);
            for (int i = 0; i < nbase; i++) std::memcpy(&hb[(size_t)i * kMaxK], pool[i].row.data(), kMaxK);
            if (cudaMemcpyAsync(base, hb.data(), hb.size(), cudaMemcpyHostToDevice, st) != cudaSuccess) { s = KO_ERR_CUDA; break; }
            if ((s = cuda_ok(ko_mlp_neighbours(base, nbase, n, nb, st)))) break;
            const int q = nbase * per, qpad = (q + 127) / 128 * 128;
            for (int off = 0; off < qpad && !s; off += C) {
                const int c = qpad - off < C ? qpad - off : C;
                if ((s = cuda_ok(ko_mlp_encode(nb + (size_t)off * kMaxK, kMaxK, tb.set_n, tb.kfeat, tb.gfeat, c,
                                               md->a0, st))))
                    break;
                if ((s = forward(md, c, false, st))) break;
                if (cudaMemcpyAsync(y_all + off, md->y, sizeof(float) * c, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                    s = KO_ERR_CUDA;
            }
            const int kk = q < k2 ? q : k2;
            if (!s) s = cuda_ok(ko_mlp_topk(y_all, q, kk, sel_state, sel_hist, sel_cnt, top_idx, st));
            if (!s) s = cuda_ok(ko_mlp_gather_rows(nb, kMaxK, top_idx, kk, top_rows, st));
            if (!s) s = exact_rows(&md->fast, tb.sets, h, 0, top_rows, kk, top_ms, d_chunk, st);
            if (!s) s = collect(kk);
        }
        // exact steepest descent from the best exact order (the simulator alone decides)
        if (!s && md->polish > 0 && !pool.empty()) {
            if (cudaStreamSynchronize(st) != cudaSuccess) s = KO_ERR_CUDA;
            std::vector<int32_t> start(n), out(n);
            for (int i = 0; i < n; i++) start[i] = pool[0].row[i];
            int64_t pms = -1, evals = 0;
            int32_t steps = 0;
            double lms = 0.0;
            if (!s) s = descend(&md->fast, h, start.data(), true, md->polish, out.data(), &pms, &steps, &evals, &lms,
                                st, polish);
            if (!s && pms >= 0 && pms < pool[0].ms) {
                pool[0].ms = pms;
                for (int i = 0; i < n; i++) pool[0].row[i] = (int8_t)out[i];
            }
        }
        cudaEventRecord(e1, st);
        if (!s && cudaStreamSynchronize(st) != cudaSuccess) s = KO_ERR_CUDA;
    }
    if (!s) s = ko_model_check(md);
    if (!s && pool.empty()) s = KO_ERR_STATE;
    if (!s) {
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (gpu_ms) *gpu_ms = ms;
        *best_makespan = pool[0].ms;
        for (int i = 0; i < n; i++) best_order[i] = pool[0].row[i];
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    return s;
}

ko_status ko_random_search_set(KoFastState *fs, const KoSet &h, long long n_orders, uint64_t seed,
                               int32_t *best_order, int64_t *best_makespan, double *gpu_ms, cudaStream_t st)
{
    if (n_orders < 1 || n_orders > (1ll << 26)) return KO_ERR_ARG;
    if (!ko_fast_applicable(h)) return KO_ERR_OVERFLOW;
    const KoSet *hs[1] = {&h};
    SetTables tb;
    ko_status s = build_tables(hs, 1, &tb, st);
    if (s) return s;
    int8_t *rows = nullptr;
    int64_t *ms = nullptr;
    KoChunk *d_chunk = nullptr;
    if (!dalloc(&rows, (size_t)n_orders * kMaxK) || !dalloc(&ms, (size_t)n_orders) || !dalloc(&d_chunk, 1))
        s = KO_ERR_NOMEM;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (!s) s = make_events(&e0, &e1);
    if (!s) {
        cudaEventRecord(e0, st);
        s = cuda_ok(ko_mlp_random_orders(rows, kMaxK, n_orders, h.n, mix64(seed ^ 0xBEEFull), st));
        if (!s) s = exact_rows(fs, tb.sets, h, 0, rows, n_orders, ms, d_chunk, st);
        cudaEventRecord(e1, st);
        if (!s && cudaStreamSynchronize(st) != cudaSuccess) s = KO_ERR_CUDA;
    }
    if (!s) {
        float t = 0.0f;
        cudaEventElapsedTime(&t, e0, e1);
        if (gpu_ms) *gpu_ms = t;
        long long bi = 0;
        s = best_of(ms, n_orders, best_makespan, &bi);
        int8_t r[kMaxK];
        if (!s && cudaMemcpy(r, rows + (size_t)bi * kMaxK, kMaxK, cudaMemcpyDeviceToHost) != cudaSuccess)
            s = KO_ERR_CUDA;
        if (!s)
            for (int i = 0; i < h.n; i++) best_order[i] = r[i];
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(rows); cudaFree(ms); cudaFree(d_chunk);
    return s;
}

// Steepest-descent hill climbing with exact scoring.  Neighbours of the
// current order are swaps of two positions, then moves of one kernel to another
// position; every one is simulated exactly, the lowest makespan wins (lowest
// neighbour index among equals) and the walk moves only on a strict improvement.
// The walk is on the device (ko_mlp_descend): an evaluation and the choice of the
// next order follow each other without the host, which looks every kAhead steps
// whether the descent has ended (the rows of an ended one are passed over).
// The start is evaluated with its neighbours.
ko_status ko_local_search_set(KoFastState *fs, const KoSet &h, const int32_t *start, bool moves, int max_iters,
                              int32_t *order_out, int64_t *makespan_out, int32_t *steps_out, int64_t *evals_out,
                              double *gpu_ms, cudaStream_t st)
{
    if (h.n < 1) return KO_ERR_ARG;
    DescentWork work;
    Carve need(nullptr);
    work.carve(need, h.n);
    ArenaUse use{fs, st};
    const ko_status s = ensure_arena(fs, need.size);
    if (s) return s;
    Carve mem(fs->arena);
    work.carve(mem, h.n);
    return descend(fs, h, start, moves, max_iters, order_out, makespan_out, steps_out, evals_out, gpu_ms, st, work);
}

static ko_status descend(KoFastState *fs, const KoSet &h, const int32_t *start, bool moves, int max_iters,
                         int32_t *order_out, int64_t *makespan_out, int32_t *steps_out, int64_t *evals_out,
                         double *gpu_ms, cudaStream_t st, const DescentWork &work)
{
    constexpr int kAhead = 3;
    const int n = h.n;
    if (n < 1 || max_iters < 0 || max_iters > (1 << 20)) return KO_ERR_ARG;
    if (!ko_fast_applicable(h)) return KO_ERR_OVERFLOW;
    KoDescent d{};
    d.makespan = -1;
    d.max_steps = max_iters;
    {
        std::vector<char> seen(n, 0);
        for (int i = 0; i < n; i++) {
            if (start[i] < 0 || start[i] >= n || seen[start[i]]) return KO_ERR_ARG;
            seen[start[i]] = 1;
            d.order[i] = (int8_t)start[i];
        }
    }
    const KoSet *hs[1] = {&h};
    SetTables tb;
    ko_status s = build_tables(hs, 1, &tb, st);
    if (s) return s;
    const int swaps = n * (n - 1) / 2, per = swaps + n * (n - 1);
    const int nq = max_iters > 0 ? (moves ? per : swaps) : 0;
    KoDescent *const state = work.state;
    int8_t *const rows = work.rows;
    int64_t *const ms = work.ms;
    KoChunk *const d_chunk = work.chunk;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if ((s = make_events(&e0, &e1))) return s;
    cudaEventRecord(e0, st);
    if (cudaMemcpyAsync(state, &d, sizeof(d), cudaMemcpyHostToDevice, st) != cudaSuccess) s = KO_ERR_CUDA;
    if (!s && nq > 0) s = cuda_ok(ko_mlp_neighbours(state->order, 1, n, rows, st));
    if (!s && cudaMemcpyAsync(rows + (size_t)nq * kMaxK, state->order, kMaxK, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        s = KO_ERR_CUDA;
    bool first = true;
    while (!s && !d.done) {
        for (int i = 0; i < kAhead && !s; i++) {
            s = exact_rows(fs, tb.sets, h, 0, rows, nq + 1, ms, d_chunk, st, first);
            first = false;
            if (!s) s = cuda_ok(ko_mlp_descend(state, ms, nq, n, rows, st));
        }
        if (!s && (cudaMemcpyAsync(&d, state, sizeof(d), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                   cudaStreamSynchronize(st) != cudaSuccess))
            s = KO_ERR_CUDA;
    }
    if (!s && d.failed) s = KO_ERR_STATE;
    cudaEventRecord(e1, st);
    if (!s && cudaStreamSynchronize(st) != cudaSuccess) s = KO_ERR_CUDA;
    if (!s) {
        float t = 0.0f;
        cudaEventElapsedTime(&t, e0, e1);
        if (gpu_ms) *gpu_ms = t;
        for (int i = 0; i < n; i++) order_out[i] = d.order[i];
        *makespan_out = d.makespan;
        if (steps_out) *steps_out = d.steps;
        if (evals_out) *evals_out = d.evals;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return s;
}

// Features of explicit orders of one set (encoder output as floats), for tests.
ko_status ko_model_features(const KoSet &h, const int8_t *orders, long long n, float *x_out, cudaStream_t st)
{
    const KoSet *hs[1] = {&h};
    SetTables tb;
    ko_status s = build_tables(hs, 1, &tb, st);
    if (s) return s;
    int8_t *rows = nullptr;
    uint16_t *x = nullptr;
    if (!dalloc(&rows, (size_t)n * kMaxK) || !dalloc(&x, (size_t)n * kMlpIn)) {
        cudaFree(rows);
        return KO_ERR_NOMEM;
    }
    std::vector<int8_t> hr((size_t)n * kMaxK, 0);
    for (long long i = 0; i < n; i++) std::memcpy(&hr[(size_t)i * kMaxK], orders + (size_t)i * h.n, h.n);
    std::vector<uint16_t> hx((size_t)n * kMlpIn);
    if (cudaMemcpyAsync(rows, hr.data(), hr.size(), cudaMemcpyHostToDevice, st) != cudaSuccess) s = KO_ERR_CUDA;
    if (!s) s = cuda_ok(ko_mlp_encode(rows, kMaxK, tb.set_n, tb.kfeat, tb.gfeat, (int)n, x, st));
    if (!s && (cudaMemcpyAsync(hx.data(), x, hx.size() * 2, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
               cudaStreamSynchronize(st) != cudaSuccess))
        s = KO_ERR_CUDA;
    if (!s)
        for (size_t i = 0; i < hx.size(); i++) {
            const uint32_t u = (uint32_t)hx[i] << 16;
            std::memcpy(&x_out[i], &u, 4);
        }
    cudaFree(rows);
    cudaFree(x);
    return s;
}

// 3D U-Net runtime: a learned initial guess for the forward solves (not in
// the paper).  Four levels (16, 32, 64, 128 channels), two 3x3x3 ReLU convs
// per level, 2x2x2 average pooling down, nearest upsampling + skip
// concatenation up, and a final linear 3x3x3 conv whose channel 0 is the
// predicted fluence.  Weights are fp32 masters with bf16 copies; every conv
// runs on the bf16 tensor-core kernels of unet_kernels.cu, forward and
// backward, and Adam updates the masters.
//
// Input features on a Kuhn grid (node index = voxel index, n a multiple of
// 8): log(mu / 0.01), log(kappa / 0.33) and the load vector of the
// illumination (2 integral Phi lambda_i, Appendix) divided by h^2; target:
// the fluence phi of that illumination.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "abi_internal.h"
#include "unet_kernels.cuh"

using bf16 = __nv_bfloat16;
using namespace qpat;

namespace {

struct Conv {
    int cin = 0, cout = 0, lvl = 0, relu = 1;
    float *w32 = nullptr, *b32 = nullptr;      // masters
    bf16 *w = nullptr, *wt = nullptr;           // bf16 copy and its flipped transpose
    float *aw = nullptr, *ab = nullptr;         // gradient summed over the samples
    float *mw = nullptr, *vw = nullptr, *mb = nullptr, *vb = nullptr;
    int64_t nw() const { return int64_t(27) * cin * cout; }
};

__global__ void k_features(int64_t nvox, const double* mu, const double* kappa, const double* f, double inv_h2,
                           float* x) {
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < nvox; v += int64_t(gridDim.x) * blockDim.x) {
        x[v * 3 + 0] = float(log(mu[v] / 0.01));
        x[v * 3 + 1] = float(log(kappa[v] / 0.33));
        x[v * 3 + 2] = float(f[v] * inv_h2);
    }
}

// network input (channels-last, 16 channels, 3 used) from fp32 features, a voxel a thread
__global__ void k_pack_input(int64_t nvox, const float* x, bf16* xin) {
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < nvox; v += int64_t(gridDim.x) * blockDim.x) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(x[3 * v], x[3 * v + 1]), b = __floats2bfloat162_rn(x[3 * v + 2], 0.f);
        uint4* o = reinterpret_cast<uint4*>(xin + v * 16);
        o[0] = make_uint4(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b), 0u, 0u);
        o[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// channel 0 of the output; in log mode (log_floor > 0) the network's output
// is log(phi) and the prediction is its exponential
__global__ void k_take_channel0(int64_t nvox, const float* y32, float* y, float log_floor) {
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < nvox; v += int64_t(gridDim.x) * blockDim.x)
        y[v] = log_floor > 0.f ? expf(y32[v * 16]) : y32[v * 16];
}

// mean-squared error of the predictions y32 and its gradient (bf16, channel 0 of 16); in
// log mode against log(max(t, log_floor))
__global__ void k_mse(int64_t nvox, const float* y32, const float* t, float scale, bf16* dy, float* loss,
                      float log_floor) {
    __shared__ float red[256];
    float s = 0.f;
    for (int64_t v = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; v < nvox; v += int64_t(gridDim.x) * blockDim.x) {
        const float tv = log_floor > 0.f ? logf(fmaxf(t[v], log_floor)) : t[v];
        const float d = y32[v] - tv;
        s += d * d;
        const __nv_bfloat162 g = __halves2bfloat162(__float2bfloat16(2.f * d * scale), __float2bfloat16(0.f));
        uint4* o = reinterpret_cast<uint4*>(dy + v * 16);
        o[0] = make_uint4(*reinterpret_cast<const uint32_t*>(&g), 0u, 0u, 0u);
        o[1] = make_uint4(0u, 0u, 0u, 0u);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0] * scale);
}

__global__ void k_f32_to_f64(int64_t n, const float* in, double* out) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        out[i] = double(in[i]);
}

int g1(int64_t n) { return int(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16))); }

}  // namespace

// Activations of a batch of samples, and what training needs beside them.
struct UnetActs {
    bf16 *xin, *a0, *s0, *p0, *a1, *s1, *p1, *a2, *s2, *p2, *a3, *bt, *a4, *d2, *a5, *d1, *a6, *d0;
};
struct UnetTrainActs {
    bf16 *cat2, *cat1, *cat0;
    bf16 *g_y, *g_d0, *g_a6, *g_cat0, *g_d1, *g_s0, *g_a5, *g_cat1, *g_d2, *g_s1, *g_a4, *g_cat2, *g_bt, *g_s2, *g_a3,
        *g_p2, *g_a2, *g_p1, *g_a1, *g_p0, *g_a0;
    float* y;        // predictions of a training batch
    float* partial;  // wgrad scratch
};

struct qpat_unet_s : UnetActs, UnetTrainActs {
    int n = 0;
    int device = 0;
    int step = 0;
    std::vector<Conv> conv;
    std::vector<void*> allocs;
    int lv[4] = {0, 0, 0, 0};  // grid side per level
    // activations (bf16 channels-last) of up to cap samples, one behind the
    // other, and (train_cap samples) the concatenations and gradients that
    // training needs; see reserve
    int cap = 0, train_cap = 0;
    int most = 0, train_most = 0;  // samples beyond which an allocation failed (0: none has)
    std::vector<void*> acts, train_acts;
    // Buffers that a captured call works on are kept for the graph's replays
    // when later calls outgrow them.
    bool acts_captured = false, train_captured = false;
    std::vector<void*> kept;
    float log_floor = 0.f;  // > 0: the network learns log(max(phi, log_floor)) (qpat_unet_set_log_output)
    float* grad = nullptr;     // every aw and ab in the order of the parameters
    float* loss = nullptr;
    float* hloss = nullptr;
};

namespace {

template <typename T>
int alloc_in(std::vector<void*>& list, T** p, size_t count) {
    void* v = nullptr;
    const cudaError_t e = cudaMalloc(&v, std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) return cuda_fail(e, "qpat_unet: cudaMalloc");
    list.push_back(v);
    *p = static_cast<T*>(v);
    return QPAT_OK;
}

template <typename T>
int ualloc(qpat_unet_s* U, T** p, size_t count) {
    const int rc = alloc_in(U->allocs, p, count);
    if (rc != QPAT_OK) return rc;
    const cudaError_t e = cudaMemset(*p, 0, std::max<size_t>(count, 1) * sizeof(T));
    return e == cudaSuccess ? QPAT_OK : cuda_fail(e, "qpat_unet: memset");
}

#define UCK(x)                                           \
    do {                                                 \
        cudaError_t e_ = (x);                            \
        if (e_ != cudaSuccess) return cuda_fail(e_, #x); \
    } while (0)

// Samples that go through the network at once: all of a call's, as far as
// their activations take at most kActBytes (at least one sample; the layers of
// a coarse level of one sample fill a few SMs only).
constexpr size_t kActBytes = size_t(8) << 30;
constexpr int kMaxSamples = 64;

// Room for up to `want` samples in place of what `list` holds (the pointers in
// P, which `each` allocates): halved where memory is short, and the room that
// there was is given up only for more.
template <typename P, typename F>
int grow(qpat_unet_s* U, std::vector<void*>& list, int& cap, int& most, bool& captured, int want, const F& each) {
    const P old = *U;
    const std::string message = g_err;
    for (; want > cap; want /= 2) {
        std::vector<void*> fresh;
        int rc = QPAT_OK;
        each([&](auto** p, size_t count) {
            if (!rc) rc = alloc_in(fresh, p, count * size_t(want));
        }, want);
        if (rc == QPAT_OK) {
            if (captured)
                U->kept.insert(U->kept.end(), list.begin(), list.end());
            else
                for (void* p : list) cudaFree(p);
            list.swap(fresh);
            captured = false;
            cap = want;
            break;
        }
        for (void* p : fresh) cudaFree(p);
        static_cast<P&>(*U) = old;
        most = std::max(cap, want / 2);
    }
    if (cap < 1) return QPAT_ECUDA;  // not even one sample's: the allocation's message stands
    g_err = message;
    return QPAT_OK;
}

// Room for min(B, what kActBytes holds) samples, also for training; kept for
// later calls and grown on demand (the device finishes its work before memory
// is released).  Where memory is short, for as many as it holds, and no more is
// tried again.  A call that is being captured into a graph can neither allocate
// nor wait: it takes the room that there is (one sample's from the start) in
// groups.
int reserve(qpat_unet_s* U, int B, bool train, cudaStream_t s) {
    const size_t v0 = size_t(U->n) * U->n * U->n, v1 = v0 / 8, v2 = v1 / 8, v3 = v2 / 8;
    const size_t fwd = 2 * (v0 * 80 + v1 * 176 + v2 * 352 + v3 * 320);
    const size_t bwd = 2 * (v0 * 176 + v1 * 352 + v2 * 704 + v3 * 320) + 4 * v0;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    const cudaError_t asked = cudaStreamIsCapturing(s, &capture);
    if (asked != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        (void)cudaGetLastError();  // another stream's capture forbids the question on the default one
        if (U->cap < 1 || U->train_cap < 1) return fail(QPAT_ECUDA, "qpat_unet: no activations, and none can be had in a capture");
        U->acts_captured = U->train_captured = true;  // the mma.sync engine's scratch lies in the training buffers
        return QPAT_OK;
    }
    auto fit = [&](size_t bytes, int most) {
        const int want = int(std::max<size_t>(1, std::min<size_t>(size_t(std::min(B, kMaxSamples)), kActBytes / bytes)));
        return most ? std::min(want, most) : want;
    };
    const int want = fit(train ? fwd + bwd : fwd, U->most);
    const int want_train = std::min(fit(fwd + bwd, U->train_most), std::max(want, U->cap));
    const bool more = want > U->cap, more_train = train && want_train > U->train_cap;
    if (!more && !more_train) return QPAT_OK;
    UCK(cudaStreamSynchronize(s));
    int rc = QPAT_OK;
    if (more)
        rc = grow<UnetActs>(U, U->acts, U->cap, U->most, U->acts_captured, want, [&](auto A, int) {
            A(&U->xin, v0 * 16); A(&U->a0, v0 * 16); A(&U->s0, v0 * 16); A(&U->p0, v1 * 16); A(&U->a1, v1 * 32);
            A(&U->s1, v1 * 32); A(&U->p1, v2 * 32); A(&U->a2, v2 * 64); A(&U->s2, v2 * 64); A(&U->p2, v3 * 64);
            A(&U->a3, v3 * 128); A(&U->bt, v3 * 128); A(&U->a4, v2 * 64); A(&U->d2, v2 * 64); A(&U->a5, v1 * 32);
            A(&U->d1, v1 * 32); A(&U->a6, v0 * 16); A(&U->d0, v0 * 16);
        });
    if (!rc && more_train)
        rc = grow<UnetTrainActs>(U, U->train_acts, U->train_cap, U->train_most, U->train_captured, want_train,
                                 [&](auto A, int samples) {
            A(&U->cat2, v2 * 192); A(&U->cat1, v1 * 96); A(&U->cat0, v0 * 48);
            A(&U->g_y, v0 * 16); A(&U->g_d0, v0 * 16); A(&U->g_a6, v0 * 16); A(&U->g_cat0, v0 * 48); A(&U->g_d1, v1 * 32);
            A(&U->g_s0, v0 * 16); A(&U->g_a5, v1 * 32); A(&U->g_cat1, v1 * 96); A(&U->g_d2, v2 * 64); A(&U->g_s1, v1 * 32);
            A(&U->g_a4, v2 * 64); A(&U->g_cat2, v2 * 192); A(&U->g_bt, v3 * 128); A(&U->g_s2, v2 * 64); A(&U->g_a3, v3 * 128);
            A(&U->g_p2, v3 * 64); A(&U->g_a2, v2 * 64); A(&U->g_p1, v2 * 32); A(&U->g_a1, v1 * 32); A(&U->g_p0, v1 * 16);
            A(&U->g_a0, v0 * 16);
            A(&U->y, v0);
            size_t scratch = 0;
            for (int b = 1; b <= samples; ++b)  // the chunking of a smaller batch may need more
                for (const Conv& c : U->conv) scratch = std::max(scratch, unet::wgrad_scratch(U->lv[c.lvl], c.cin, c.cout, b));
            A(&U->partial, (scratch + samples - 1) / samples);
        });
    return rc;
}

// One convolution of B samples.  On the tcgen05 engine one launch, which reads
// a concatenation from its two parts; the mma.sync engine goes sample by
// sample through materialised tensors.
int conv_fwd(qpat_unet_s* U, const bf16* w, int Cout, const float* bias, int relu,
             const unet::ConvInput& in, const unet::ConvOutput& out, int n, int B, cudaStream_t s) {
    const int Cin = in.Clo + in.Cskip;
    if (unet::conv_engine() == 0 && unet::conv3d_fwd_tc_supported(Cin, Cout)) {
        UCK(unet::conv3d_fwd_tc(in, w, bias, Cout, relu, out, n, B, s));
        return QPAT_OK;
    }
    // one sample's concatenation and last layer, in training buffers that are free here: training writes its
    // concatenations itself, and the gradients of the output and of cat0 after the forward pass
    bf16 *const cat = U->cat0, *const last = U->g_y;
    float* const last32 = reinterpret_cast<float*>(U->g_cat0);
    const int64_t nv = int64_t(n) * n * n;
    for (int b = 0; b < B; ++b) {
        const bf16* x = in.skip + b * nv * in.Cskip;
        if (in.lo) {
            UCK(unet::upcat(in.lo + b * (nv / 8) * in.Clo, in.Clo, x, in.Cskip, n, 1, cat, s));
            x = cat;
        }
        UCK(unet::conv3d_fwd(x, Cin, w, bias, Cout, relu, out.bf ? out.bf + b * nv * Cout : last,
                             out.first ? last32 : out.f32, n, s));
        if (out.first) {
            qpat::note_launch(1);
            k_take_channel0<<<g1(nv), 256, 0, s>>>(nv, last32, out.first + b * nv, out.first_exp ? 1.f : 0.f);
        }
    }
    return QPAT_OK;
}

int conv_fwd(qpat_unet_s* U, const Conv& c, const unet::ConvInput& in, bf16* out, int n, int B, cudaStream_t s) {
    return conv_fwd(U, c.w, c.cout, c.b32, c.relu, in, unet::ConvOutput{out}, n, B, s);
}

// backward of one conv: gout (gradient of its output, masked here by the
// ReLU through `out`) -> weight/bias gradient (added to what is there when
// add is set), and gin if not null
int conv_bwd(qpat_unet_s* U, Conv& c, const bf16* in, const bf16* out, bf16* gout, bf16* gin, int n, int B, int add,
             cudaStream_t s) {
    const int64_t nv = int64_t(n) * n * n * B;
    if (c.relu) UCK(unet::relu_mask(gout, out, nv * c.cout, s));
    UCK(unet::conv3d_wgrad(in, c.cin, gout, c.cout, c.aw, c.ab, U->partial, n, B, add, s));
    if (gin) return conv_fwd(U, c.wt, c.cin, nullptr, 0, unet::ConvInput{gout, c.cout}, unet::ConvOutput{gin}, n, B, s);
    return QPAT_OK;
}

// The network on B samples in xin; y (B n^3 floats) receives channel 0 of the
// last layer (y_exp: its exponential).  train: the concatenations are also
// written out for the backward pass.
int unet_forward(qpat_unet_s* U, int B, bool train, float* y, int y_exp, cudaStream_t s) {
    auto& C = U->conv;
    using In = unet::ConvInput;
    const int n0 = U->lv[0], n1 = U->lv[1], n2 = U->lv[2], n3 = U->lv[3];
    int rc;
    if ((rc = conv_fwd(U, C[0], In{U->xin, 16}, U->a0, n0, B, s)) || (rc = conv_fwd(U, C[1], In{U->a0, 16}, U->s0, n0, B, s)))
        return rc;
    UCK(unet::avgpool(U->s0, 16, n0, B, U->p0, s));
    if ((rc = conv_fwd(U, C[2], In{U->p0, 16}, U->a1, n1, B, s)) || (rc = conv_fwd(U, C[3], In{U->a1, 32}, U->s1, n1, B, s)))
        return rc;
    UCK(unet::avgpool(U->s1, 32, n1, B, U->p1, s));
    if ((rc = conv_fwd(U, C[4], In{U->p1, 32}, U->a2, n2, B, s)) || (rc = conv_fwd(U, C[5], In{U->a2, 64}, U->s2, n2, B, s)))
        return rc;
    UCK(unet::avgpool(U->s2, 64, n2, B, U->p2, s));
    if ((rc = conv_fwd(U, C[6], In{U->p2, 64}, U->a3, n3, B, s)) || (rc = conv_fwd(U, C[7], In{U->a3, 128}, U->bt, n3, B, s)))
        return rc;
    auto cat = [&](const bf16* lo, int clo, const bf16* skip, int cs, int n, bf16* to, In& in) -> cudaError_t {
        in = train ? In{to, clo + cs} : In{skip, cs, lo, clo};
        return train ? unet::upcat(lo, clo, skip, cs, n, B, to, s) : cudaSuccess;
    };
    In in{};
    UCK(cat(U->bt, 128, U->s2, 64, n2, U->cat2, in));
    if ((rc = conv_fwd(U, C[8], in, U->a4, n2, B, s)) || (rc = conv_fwd(U, C[9], In{U->a4, 64}, U->d2, n2, B, s))) return rc;
    UCK(cat(U->d2, 64, U->s1, 32, n1, U->cat1, in));
    if ((rc = conv_fwd(U, C[10], in, U->a5, n1, B, s)) || (rc = conv_fwd(U, C[11], In{U->a5, 32}, U->d1, n1, B, s))) return rc;
    UCK(cat(U->d1, 32, U->s0, 16, n0, U->cat0, in));
    if ((rc = conv_fwd(U, C[12], in, U->a6, n0, B, s)) || (rc = conv_fwd(U, C[13], In{U->a6, 16}, U->d0, n0, B, s))) return rc;
    unet::ConvOutput out;
    out.first = y;
    out.first_exp = y_exp;
    return conv_fwd(U, C[14].w, 16, C[14].b32, 0, In{U->d0, 16}, out, n0, B, s);
}

int unet_backward(qpat_unet_s* U, int B, int add, cudaStream_t s) {
    auto& C = U->conv;
    const int n0 = U->lv[0], n1 = U->lv[1], n2 = U->lv[2], n3 = U->lv[3];
    int rc;
    auto bwd = [&](int i, const bf16* in, const bf16* out, bf16* gout, bf16* gin, int n) {
        return rc = conv_bwd(U, C[size_t(i)], in, out, gout, gin, n, B, add, s);
    };
    if (bwd(14, U->d0, nullptr, U->g_y, U->g_d0, n0) || bwd(13, U->a6, U->d0, U->g_d0, U->g_a6, n0) ||
        bwd(12, U->cat0, U->a6, U->g_a6, U->g_cat0, n0))
        return rc;
    UCK(unet::upcat_bwd(U->g_cat0, 32, 16, n0, B, U->g_d1, U->g_s0, 0, s));
    if (bwd(11, U->a5, U->d1, U->g_d1, U->g_a5, n1) || bwd(10, U->cat1, U->a5, U->g_a5, U->g_cat1, n1)) return rc;
    UCK(unet::upcat_bwd(U->g_cat1, 64, 32, n1, B, U->g_d2, U->g_s1, 0, s));
    if (bwd(9, U->a4, U->d2, U->g_d2, U->g_a4, n2) || bwd(8, U->cat2, U->a4, U->g_a4, U->g_cat2, n2)) return rc;
    UCK(unet::upcat_bwd(U->g_cat2, 128, 64, n2, B, U->g_bt, U->g_s2, 0, s));
    if (bwd(7, U->a3, U->bt, U->g_bt, U->g_a3, n3) || bwd(6, U->p2, U->a3, U->g_a3, U->g_p2, n3)) return rc;
    UCK(unet::avgpool_bwd(U->g_p2, 64, n2, B, U->g_s2, 1, s));
    if (bwd(5, U->a2, U->s2, U->g_s2, U->g_a2, n2) || bwd(4, U->p1, U->a2, U->g_a2, U->g_p1, n2)) return rc;
    UCK(unet::avgpool_bwd(U->g_p1, 32, n1, B, U->g_s1, 1, s));
    if (bwd(3, U->a1, U->s1, U->g_s1, U->g_a1, n1) || bwd(2, U->p0, U->a1, U->g_a1, U->g_p0, n1)) return rc;
    UCK(unet::avgpool_bwd(U->g_p0, 16, n0, B, U->g_s0, 1, s));
    if (bwd(1, U->a0, U->s0, U->g_s0, U->g_a0, n0) || bwd(0, U->xin, U->a0, U->g_a0, nullptr, n0)) return rc;
    return QPAT_OK;
}

int refresh_bf16(qpat_unet_s* U, cudaStream_t s) {
    for (auto& c : U->conv) {
        UCK(unet::f32_to_bf16(c.w32, c.w, c.nw(), s));
        UCK(unet::flip_weights(c.w, c.cin, c.cout, c.wt, s));
    }
    return QPAT_OK;
}

}  // namespace

extern "C" {

int qpat_unet_create(int n, uint64_t seed, qpat_unet_t* out) {
    if (!out) return fail(QPAT_EINVAL, "qpat_unet_create: out is NULL");
    *out = nullptr;
    if (n < 32 || n % 16 || n > 512)
        return fail(QPAT_EINVAL, "qpat_unet_create: n must be a multiple of 16 in [32, 512]");
    auto* U = new qpat_unet_s();
    cudaGetDevice(&U->device);
    U->n = n;
    for (int l = 0; l < 4; ++l) U->lv[l] = n >> l;
    // (cin, cout, level, relu) of the 15 convs
    const int spec[15][4] = {{16, 16, 0, 1},  {16, 16, 0, 1},  {16, 32, 1, 1},  {32, 32, 1, 1},  {32, 64, 2, 1},
                             {64, 64, 2, 1},  {64, 128, 3, 1}, {128, 128, 3, 1}, {192, 64, 2, 1}, {64, 64, 2, 1},
                             {96, 32, 1, 1},  {32, 32, 1, 1},  {48, 16, 0, 1},  {16, 16, 0, 1},  {16, 16, 0, 0}};
    std::mt19937_64 rng(seed);
    int rc = QPAT_OK;
    for (int i = 0; i < 15 && rc == QPAT_OK; ++i) {
        Conv c;
        c.cin = spec[i][0];
        c.cout = spec[i][1];
        c.lvl = spec[i][2];
        c.relu = spec[i][3];
        const int64_t nw = c.nw();
        if ((rc = ualloc(U, &c.w32, nw)) || (rc = ualloc(U, &c.b32, c.cout)) || (rc = ualloc(U, &c.w, nw)) ||
            (rc = ualloc(U, &c.wt, nw)) || (rc = ualloc(U, &c.mw, nw)) || (rc = ualloc(U, &c.vw, nw)) || (rc = ualloc(U, &c.mb, c.cout)) || (rc = ualloc(U, &c.vb, c.cout)))
            break;
        // He-normal initialisation over the real fan-in (the first conv sees 3 channels)
        const int fan = 27 * (i == 0 ? 3 : c.cin);
        std::normal_distribution<float> nd(0.f, std::sqrt(2.f / float(fan)) * (c.relu ? 1.f : 0.5f));
        std::vector<float> hw(nw);
        for (int64_t k = 0; k < nw; ++k) {
            const int ci = int(k % c.cin);
            hw[k] = (i == 0 && ci >= 3) ? 0.f : nd(rng);
        }
        if (cudaMemcpy(c.w32, hw.data(), nw * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess)
            rc = cuda_fail(cudaGetLastError(), "qpat_unet_create: upload");
        U->conv.push_back(c);
    }
    size_t total = 0;
    for (const Conv& c : U->conv) total += size_t(c.nw()) + c.cout;
    if (!rc) rc = ualloc(U, &U->grad, total);
    if (!rc) {
        float* g = U->grad;
        for (Conv& c : U->conv) {
            c.aw = g;
            c.ab = g + c.nw();
            g = c.ab + c.cout;
        }
        rc = reserve(U, 1, true, nullptr);
    }
    if (!rc) rc = ualloc(U, &U->loss, 1);
    if (!rc && cudaMallocHost(&U->hloss, sizeof(float)) != cudaSuccess) rc = fail(QPAT_ECUDA, "qpat_unet: pinned");
    if (!rc) rc = refresh_bf16(U, nullptr);
    if (!rc && cudaDeviceSynchronize() != cudaSuccess) rc = cuda_fail(cudaGetLastError(), "qpat_unet_create");
    if (rc) {
        qpat_unet_free(U);
        return rc;
    }
    *out = U;
    return QPAT_OK;
}

void qpat_unet_free(qpat_unet_t U) {
    if (!U) return;
    DeviceGuard dg(U->device);
    cudaDeviceSynchronize();
    for (auto* list : {&U->allocs, &U->acts, &U->train_acts, &U->kept})
        for (void* p : *list) cudaFree(p);
    if (U->hloss) cudaFreeHost(U->hloss);
    delete U;
}

int64_t qpat_unet_num_params(qpat_unet_t U) {
    if (!U) return -1;
    int64_t n = 0;
    for (auto& c : U->conv) n += c.nw() + c.cout;
    return n;
}

int qpat_unet_get_params(qpat_unet_t U, float* host) {
    if (!U || !host) return fail(QPAT_EINVAL, "qpat_unet_get_params: NULL argument");
    DeviceGuard dg(U->device);
    for (auto& c : U->conv) {
        UCK(cudaMemcpy(host, c.w32, c.nw() * sizeof(float), cudaMemcpyDeviceToHost));
        host += c.nw();
        UCK(cudaMemcpy(host, c.b32, c.cout * sizeof(float), cudaMemcpyDeviceToHost));
        host += c.cout;
    }
    return QPAT_OK;
}

int qpat_unet_set_params(qpat_unet_t U, const float* host) {
    if (!U || !host) return fail(QPAT_EINVAL, "qpat_unet_set_params: NULL argument");
    DeviceGuard dg(U->device);
    for (auto& c : U->conv) {
        UCK(cudaMemcpy(c.w32, host, c.nw() * sizeof(float), cudaMemcpyHostToDevice));
        host += c.nw();
        UCK(cudaMemcpy(c.b32, host, c.cout * sizeof(float), cudaMemcpyHostToDevice));
        host += c.cout;
    }
    int rc = refresh_bf16(U, nullptr);
    if (rc) return rc;
    UCK(cudaDeviceSynchronize());
    return QPAT_OK;
}

int qpat_unet_predict_dev(qpat_unet_t U, const float* x, int B, float* y, void* stream) {
    if (!U || !x || !y || B < 1) return fail(QPAT_EINVAL, "qpat_unet_predict_dev: bad argument");
    DeviceGuard dg(U->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t nv = int64_t(U->n) * U->n * U->n;
    int rc = reserve(U, B, false, s);
    if (rc) return rc;
    for (int b = 0; b < B; b += U->cap) {
        const int nb = std::min(U->cap, B - b);
        qpat::note_launch(1);
        k_pack_input<<<g1(nv * nb), 256, 0, s>>>(nv * nb, x + b * nv * 3, U->xin);
        if ((rc = unet_forward(U, nb, false, y + b * nv, U->log_floor > 0.f, s))) return rc;
    }
    UCK(cudaGetLastError());
    return QPAT_OK;
}

// Loss (mean squared error over the B samples' voxels) into U->loss and its
// gradient with respect to every weight and bias into the accumulators
// aw, ab (summed over the samples).
static int unet_loss_grad(qpat_unet_s* U, const float* x, const float* t, int B, cudaStream_t s) {
    const int64_t nv = int64_t(U->n) * U->n * U->n;
    int rc = reserve(U, B, true, s);
    if (rc) return rc;
    UCK(cudaMemsetAsync(U->loss, 0, sizeof(float), s));
    const int cap = std::min(U->cap, U->train_cap);
    for (int b = 0; b < B; b += cap) {
        const int nb = std::min(cap, B - b);
        qpat::note_launch(1);
        k_pack_input<<<g1(nv * nb), 256, 0, s>>>(nv * nb, x + b * nv * 3, U->xin);
        if ((rc = unet_forward(U, nb, true, U->y, 0, s))) return rc;
        qpat::note_launch(1);
        k_mse<<<g1(nv * nb), 256, 0, s>>>(nv * nb, U->y, t + b * nv, 1.f / float(nv * B), U->g_y, U->loss, U->log_floor);
        if ((rc = unet_backward(U, nb, b > 0, s))) return rc;
    }
    UCK(cudaGetLastError());
    return QPAT_OK;
}

int qpat_unet_grad_dev(qpat_unet_t U, const float* x, const float* t, int B, float* grad, float* loss,
                       void* stream) {
    if (!U || !x || !t || !grad || B < 1) return fail(QPAT_EINVAL, "qpat_unet_grad_dev: bad argument");
    DeviceGuard dg(U->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = unet_loss_grad(U, x, t, B, s);
    if (rc) return rc;
    UCK(cudaMemcpyAsync(grad, U->grad, sizeof(float) * size_t(qpat_unet_num_params(U)), cudaMemcpyDeviceToHost, s));
    UCK(cudaMemcpyAsync(U->hloss, U->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
    UCK(cudaStreamSynchronize(s));
    if (loss) *loss = *U->hloss;
    return QPAT_OK;
}

int qpat_unet_set_log_output(qpat_unet_t U, double floor) {
    if (!U || !(floor >= 0.0) || !std::isfinite(floor))
        return fail(QPAT_EINVAL, "qpat_unet_set_log_output: NULL network or bad floor");
    U->log_floor = float(floor);
    return QPAT_OK;
}

int qpat_unet_train_dev(qpat_unet_t U, const float* x, const float* t, int B, float lr, float* loss, void* stream) {
    if (!U || !x || !t || B < 1) return fail(QPAT_EINVAL, "qpat_unet_train_dev: bad argument");
    DeviceGuard dg(U->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc0 = unet_loss_grad(U, x, t, B, s);
    if (rc0) return rc0;
    ++U->step;
    for (auto& c : U->conv) {
        UCK(unet::adam(c.w32, nullptr, c.aw, c.mw, c.vw, c.nw(), lr, 0.9f, 0.999f, 1e-8f, U->step, s));
        UCK(unet::adam(c.b32, nullptr, c.ab, c.mb, c.vb, c.cout, lr, 0.9f, 0.999f, 1e-8f, U->step, s));
    }
    int rc = refresh_bf16(U, s);
    if (rc) return rc;
    if (loss) {
        UCK(cudaMemcpyAsync(U->hloss, U->loss, sizeof(float), cudaMemcpyDeviceToHost, s));
        UCK(cudaStreamSynchronize(s));
        *loss = *U->hloss;
    }
    return QPAT_OK;
}

// Network input of illumination k for every illumination of a Kuhn-grid mesh
// (caller node index = voxel index): x is K x N x 3 float
int qpat_unet_features_dev(qpat_mesh_t M, const double* kappa, const double* mu, int K, const double* flux_face,
                           double h, float* x, void* stream) {
    if (!M || !kappa || !mu || !flux_face || !x || K < 1 || !(h > 0))
        return fail(QPAT_EINVAL, "qpat_unet_features_dev: bad argument");
    DeviceGuard dg(M->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t N = M->h.N;
    const int R = round_rhs(K);
    if (R < 0) return fail(QPAT_EINVAL, "qpat_unet_features_dev: K must be in [1, 16]");
    cudaError_t e = cudaSuccess;
    double* f = M->ws.get<double>("un.f", N * R, s, &e);
    double* fc = M->ws.get<double>("un.fc", N * K, s, &e);
    if (e != cudaSuccess) return cuda_fail(e, "workspace");
    UCK(cudaMemsetAsync(f, 0, N * R * sizeof(double), s));
    UCK(launch_load(M->d, K, R, flux_face, f, s));
    UCK((launch_from_lib<double, double>(M->d, K, R, f, fc, s)));
    qpat::note_launch(K);
    for (int k = 0; k < K; ++k) k_features<<<g1(N), 256, 0, s>>>(N, mu, kappa, fc + k * N, 1.0 / (h * h), x + k * N * 3);
    UCK(cudaGetLastError());
    return QPAT_OK;
}

// float predictions -> double initial guess
int qpat_unet_to_double_dev(const float* y, int64_t count, double* out, void* stream) {
    qpat::note_launch(1);
    k_f32_to_f64<<<g1(count), 256, 0, static_cast<cudaStream_t>(stream)>>>(count, y, out);
    UCK(cudaGetLastError());
    return QPAT_OK;
}

// low-level entry points of the bf16 tensor-core convolution (tests)
int qpat_conv3d_bf16_dev(const void* in, int Cin, const void* w, const float* bias, int Cout, int relu, int n,
                         void* out, float* out_f32, void* stream) {
    if (!in || !w || !out) return fail(QPAT_EINVAL, "qpat_conv3d_bf16_dev: NULL argument");
    UCK(unet::conv3d_fwd(static_cast<const bf16*>(in), Cin, static_cast<const bf16*>(w), bias, Cout, relu,
                         static_cast<bf16*>(out), out_f32, n, static_cast<cudaStream_t>(stream)));
    return QPAT_OK;
}

int qpat_conv3d_bf16_wgrad_dev(const void* in, int Cin, const void* dy, int Cout, int n, float* dw, float* db,
                               float* partial, void* stream) {
    if (!in || !dy || !dw || !partial) return fail(QPAT_EINVAL, "qpat_conv3d_bf16_wgrad_dev: NULL argument");
    UCK(unet::conv3d_wgrad(static_cast<const bf16*>(in), Cin, static_cast<const bf16*>(dy), Cout, dw, db, partial, n, 1, 0,
                           static_cast<cudaStream_t>(stream)));
    return QPAT_OK;
}

int qpat_conv3d_set_engine(int engine) {
    if (engine != 0 && engine != 1) return fail(QPAT_EINVAL, "qpat_conv3d_set_engine: engine must be 0 or 1");
    unet::set_conv_engine(engine);
    return QPAT_OK;
}

int qpat_conv3d_tc_timeouts(void) { return unet::tc_timeouts(); }

int64_t qpat_conv3d_bf16_wgrad_scratch(int n, int Cin, int Cout) {
    return int64_t(unet::wgrad_scratch(n, Cin, Cout, 1));
}

}  // extern "C"

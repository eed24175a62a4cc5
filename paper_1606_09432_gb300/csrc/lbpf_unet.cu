// The learned surrogate's network runtime: a 2D U-Net of `levels` levels
// with base * 2^l channels at level l (default 3 levels, base 16: 16, 32, 64
// channels), two periodic 3x3 convolutions + ReLU per level on the way down
// (2x2 average pooling between levels) and on the way up (nearest 2x
// upsampling concatenated with the level's skip), and a 1x1 head.
// Input per site: (phi, u, cos 4 theta, sin 4 theta, eps) zero-padded to 16
// channels; output: (d phi, d u), the change of phi and u over the jump, the
// phi channel gated by (1 - phi^2) so that the bulk phases stay untouched.
// Forward, hand-written backward and Adam run in the kernels of lbpf_nn.cu
// (3x3 convolutions and their weight gradients on the tensor cores).
#include <cmath>
#include <cstring>
#include <string>
#include <utility>
#include <vector>

#include "../../include/lbpf.h"
#include "lbpf_nn.cuh"

using namespace lbpf_nn;

namespace {

constexpr int kIn = 5;      // input channels before padding
constexpr int kInPad = 16;  // padded input channels
constexpr int kOut = 2;

struct Conv {
    int cin, cout;
    long long off_w, off_b;  // offsets in the flat FP32 parameter vector
    __nv_bfloat16* wb = nullptr;   // BF16 copy [tap][cout][cin]
    __nv_bfloat16* wt = nullptr;   // flipped BF16 weights for the data gradient
    float* part = nullptr;         // partial sums of the bias gradient
};

}  // namespace

struct lbpf_net {
    int H = 0, W = 0, N = 0, levels = 3, base = 16;
    cudaStream_t stream = nullptr;
    std::vector<Conv> conv;  // 4 levels - 2 3x3 convolutions: encoder level by level, then decoder top-down
    long long off_hw = 0, off_hb = 0, n_params = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // FP32 params, grads, Adam moments
    __nv_bfloat16* pb = nullptr;  // BF16 copies of the 3x3 weights and their flipped forms
    int adam_t = 0;
    float loss_alpha = 0.f;  // interface weight of the training loss
    // activations (N, H >> l, W >> l, c) per level l: encoder convolution
    // outputs ea, e; pooled input pl (l >= 1); decoder outputs da, d (l <
    // levels - 1; the concatenation of the upsampled level below and the skip is
    // read in its two parts)
    float *xin = nullptr, *out = nullptr;
    std::vector<float*> ea, e, pl, da, d;
    // gradient scratch per level (two of the level's widest channel count)
    std::vector<float*> ga, gb;
    float* g_out = nullptr;
    // partial sums of the head's gradients (and the last layer's bias), and the
    // table by which they and the layers' are added up
    float* head_part = nullptr;
    PartialSums sums{};
    double* d_loss = nullptr;
    std::vector<void*> allocs;
    std::string err;

    int ch(int l) const { return base << l; }
    float* top() const { return levels > 1 ? d[0] : e[0]; }
    // output of the level below decoder level l
    float* below(int l) const { return l == levels - 2 ? e[l + 1] : d[l + 1]; }
};

namespace {

thread_local std::string t_net_err;

int net_fail(lbpf_net* n, int code, const char* msg)
{
    if (n)
        n->err = msg;
    else
        t_net_err = msg;
    return code;
}

#define NK(call)                                                                                       \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess) return net_fail(net, LBPF_ECUDA, cudaGetErrorString(e_));               \
    } while (0)

float* alloc_f(lbpf_net* net, long long n)
{
    void* p = nullptr;
    if (cudaMalloc(&p, sizeof(float) * (size_t)(n > 0 ? n : 1)) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    net->allocs.push_back(p);
    cudaMemsetAsync(p, 0, sizeof(float) * (size_t)(n > 0 ? n : 1), net->stream);
    return static_cast<float*>(p);
}

// SplitMix64 for the weight initialisation.
struct Mix {
    unsigned long long s;
    unsigned long long next()
    {
        s += 0x9E3779B97F4A7C15ULL;
        unsigned long long z = s;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
        return z ^ (z >> 31);
    }
    double uniform() { return (next() >> 11) * (1.0 / 9007199254740992.0); }
};

int refresh_bf16(lbpf_net* net)
{
    for (Conv& c : net->conv) {
        NK(to_bf16(net->p + c.off_w, c.wb, 9LL * c.cin * c.cout, net->stream));
        NK(flip_weights(c.wb, c.wt, c.cin, c.cout, net->stream));
    }
    return LBPF_OK;
}

}  // namespace

extern "C" int lbpf_net_create_arch(int H, int W, int batch, int levels, int base, unsigned long long seed,
                                    void* stream, lbpf_net** out)
{
    if (!out) return net_fail(nullptr, LBPF_EINVAL, "lbpf_net_create: out is NULL");
    *out = nullptr;
    if (levels < 2 || levels > 5 || !(base == 16 || base == 32 || base == 64) || (base << (levels - 1)) > 256)
        return net_fail(nullptr, LBPF_EINVAL,
                        "lbpf_net_create: levels 2..5, base 16, 32 or 64, at most 256 channels at the deepest level");
    const int q = 8 << (levels - 1);
    if (H < q || W < q || H % q || W % q || batch < 1)
        return net_fail(nullptr, LBPF_EINVAL, "lbpf_net_create: H, W must be multiples of 8 * 2^(levels - 1), batch >= 1");
    lbpf_net* net = new (std::nothrow) lbpf_net();
    if (!net) return net_fail(nullptr, LBPF_ENOMEM, "lbpf_net_create: out of host memory");
    net->H = H;
    net->W = W;
    net->N = batch;
    net->levels = levels;
    net->base = base;
    net->stream = static_cast<cudaStream_t>(stream);
    std::vector<std::pair<int, int>> cfg = {{kInPad, net->ch(0)}, {net->ch(0), net->ch(0)}};
    for (int l = 1; l < levels; ++l) {
        cfg.push_back({net->ch(l - 1), net->ch(l)});
        cfg.push_back({net->ch(l), net->ch(l)});
    }
    for (int l = levels - 2; l >= 0; --l) {
        cfg.push_back({net->ch(l + 1) + net->ch(l), net->ch(l)});
        cfg.push_back({net->ch(l), net->ch(l)});
    }
    long long off = 0, wtot = 0;
    for (auto& c2 : cfg) {
        Conv c;
        c.cin = c2.first;
        c.cout = c2.second;
        c.off_w = off;
        off += 9LL * c.cin * c.cout;
        wtot += 9LL * c.cin * c.cout;
        c.off_b = off;
        off += c.cout;
        net->conv.push_back(c);
    }
    net->off_hw = off;
    off += kOut * net->ch(0);
    net->off_hb = off;
    off += kOut;
    net->n_params = off;

    bool ok = (net->p = alloc_f(net, off)) && (net->g = alloc_f(net, off)) && (net->m = alloc_f(net, off)) &&
              (net->v = alloc_f(net, off));
    void* pb = nullptr;
    ok = ok && cudaMalloc(&pb, sizeof(__nv_bfloat16) * (size_t)wtot * 2) == cudaSuccess;
    if (pb) net->allocs.push_back(pb);
    if (ok) {
        net->pb = static_cast<__nv_bfloat16*>(pb);
        __nv_bfloat16* cur = net->pb;
        for (Conv& c : net->conv) {
            c.wb = cur;
            cur += 9LL * c.cin * c.cout;
            c.wt = cur;
            cur += 9LL * c.cin * c.cout;
        }
    }
    const long long P0 = (long long)batch * H * W;
    net->ea.assign(levels, nullptr);
    net->e.assign(levels, nullptr);
    net->pl.assign(levels, nullptr);
    net->da.assign(levels, nullptr);
    net->d.assign(levels, nullptr);
    net->ga.assign(levels, nullptr);
    net->gb.assign(levels, nullptr);
    ok = ok && (net->xin = alloc_f(net, P0 * kInPad)) && (net->out = alloc_f(net, P0 * kOut)) &&
         (net->g_out = alloc_f(net, P0 * kOut));
    for (int l = 0; l < levels && ok; ++l) {
        const long long Pl = P0 >> (2 * l);
        const int c = net->ch(l), cw = l + 1 < levels ? c + net->ch(l + 1) : c;
        ok = (net->ea[l] = alloc_f(net, Pl * c)) && (net->e[l] = alloc_f(net, Pl * c)) &&
             (net->ga[l] = alloc_f(net, Pl * cw)) && (net->gb[l] = alloc_f(net, Pl * cw));
        if (ok && l > 0) ok = (net->pl[l] = alloc_f(net, Pl * net->ch(l - 1))) != nullptr;
        if (ok && l + 1 < levels)
            ok = (net->da[l] = alloc_f(net, Pl * c)) && (net->d[l] = alloc_f(net, Pl * c));
    }
    // level of conv k: pairs down the encoder, then pairs up the decoder
    auto level = [&](int k) { return k < 2 * levels ? k / 2 : 2 * levels - 2 - k / 2; };
    const int nc = (int)net->conv.size(), c0 = net->ch(0), hb = act_blocks(P0, c0);
    ok = ok && (net->head_part = alloc_f(net, (long long)hb * (3 * c0 + 2)));
    for (int k = 0; k + 1 < nc && ok; ++k) {
        Conv& c = net->conv[k];
        const int rows = act_blocks(P0 >> (2 * level(k)), c.cout);
        ok = (c.part = alloc_f(net, (long long)rows * c.cout)) != nullptr;
        net->sums.s[net->sums.n++] = {c.part, net->g + c.off_b, rows, c.cout, c.cout};
    }
    net->sums.s[net->sums.n++] = {net->head_part, net->g + net->off_hw, hb, 3 * c0 + 2, 2 * c0 + 2};
    net->sums.s[net->sums.n++] = {net->head_part + 2 * c0 + 2, net->g + net->conv[nc - 1].off_b, hb, 3 * c0 + 2, c0};
    void* dl = nullptr;
    ok = ok && cudaMalloc(&dl, sizeof(double)) == cudaSuccess;
    if (dl) {
        net->allocs.push_back(dl);
        net->d_loss = static_cast<double*>(dl);
    }
    if (!ok) {
        cudaGetLastError();
        for (void* q2 : net->allocs) cudaFree(q2);
        delete net;
        return net_fail(nullptr, LBPF_ENOMEM, "lbpf_net_create: device allocation failed");
    }
    // He-uniform initialisation of the 3x3 and 1x1 weights, zero biases.
    std::vector<float> h((size_t)off, 0.f);
    Mix rng{seed};
    for (const Conv& c : net->conv) {
        const double a = std::sqrt(6.0 / (9.0 * c.cin));
        for (long long k = 0; k < 9LL * c.cin * c.cout; ++k) h[c.off_w + k] = (float)((2 * rng.uniform() - 1) * a);
    }
    for (int k = 0; k < kOut * net->ch(0); ++k) h[net->off_hw + k] = (float)((2 * rng.uniform() - 1) * 1e-2);
    if (cudaMemcpyAsync(net->p, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice, net->stream) !=
            cudaSuccess ||
        refresh_bf16(net) != LBPF_OK || cudaStreamSynchronize(net->stream) != cudaSuccess) {
        cudaGetLastError();
        for (void* q2 : net->allocs) cudaFree(q2);
        delete net;
        return net_fail(nullptr, LBPF_ECUDA, "lbpf_net_create: initialisation failed");
    }
    *out = net;
    return LBPF_OK;
}

extern "C" int lbpf_net_create(int H, int W, int batch, unsigned long long seed, void* stream, lbpf_net** out)
{
    return lbpf_net_create_arch(H, W, batch, 3, 16, seed, stream, out);
}

extern "C" int lbpf_net_destroy(lbpf_net* net)
{
    if (!net) return LBPF_OK;
    cudaStreamSynchronize(net->stream);
    for (void* q : net->allocs) cudaFree(q);
    delete net;
    return LBPF_OK;
}

extern "C" const char* lbpf_net_last_error(const lbpf_net* net) { return net ? net->err.c_str() : t_net_err.c_str(); }

extern "C" int lbpf_net_num_params(const lbpf_net* net, long long* n)
{
    if (!net || !n) return LBPF_EINVAL;
    *n = net->n_params;
    return LBPF_OK;
}

extern "C" int lbpf_net_get_params(lbpf_net* net, float* host, int which)
{
    if (!net || !host) return LBPF_EINVAL;
    const float* src = which == 1 ? net->g : net->p;
    NK(cudaMemcpyAsync(host, src, sizeof(float) * net->n_params, cudaMemcpyDeviceToHost, net->stream));
    NK(cudaStreamSynchronize(net->stream));
    return LBPF_OK;
}

extern "C" int lbpf_net_set_params(lbpf_net* net, const float* host)
{
    if (!net || !host) return LBPF_EINVAL;
    NK(cudaMemcpyAsync(net->p, host, sizeof(float) * net->n_params, cudaMemcpyHostToDevice, net->stream));
    int rc = refresh_bf16(net);
    if (rc) return rc;
    NK(cudaStreamSynchronize(net->stream));
    return LBPF_OK;
}

namespace {

int forward(lbpf_net* net, const float* x, float* y)
{
    const int N = net->N, H = net->H, W = net->W, lv = net->levels;
    const long long P0 = (long long)N * H * W;
    cudaStream_t s = net->stream;
    auto cv = [&](int k, const float* in, float* o, int l) -> cudaError_t {
        const Conv& c = net->conv[k];
        return conv3x3_fwd(in, c.wb, net->p + c.off_b, o, N, H >> l, W >> l, c.cin, c.cout, 1, s);
    };
    NK(pad_channels(x, net->xin, P0, kIn, kInPad, s));
    int k = 0;
    for (int l = 0; l < lv; ++l) {
        const float* a = net->xin;
        if (l > 0) {
            NK(pool_fwd(net->e[l - 1], net->pl[l], N, H >> (l - 1), W >> (l - 1), net->ch(l - 1), s));
            a = net->pl[l];
        }
        NK(cv(k, a, net->ea[l], l));
        NK(cv(k + 1, net->ea[l], net->e[l], l));
        k += 2;
    }
    for (int l = lv - 2; l >= 0; --l) {
        const Conv& c = net->conv[k];
        NK(conv3x3_fwd_src(net->below(l), net->e[l], net->ch(l + 1), net->ch(l), c.wb, net->p + c.off_b, net->da[l], N,
                           H >> l, W >> l, c.cout, 1, s));
        NK(cv(k + 1, net->da[l], net->d[l], l));
        k += 2;
    }
    NK(head_fwd(net->top(), net->p + net->off_hw, net->p + net->off_hb, net->xin, kInPad, net->out, y, P0, net->ch(0),
                s));
    return LBPF_OK;
}

// Backward from dy (dL/d out); accumulates parameter gradients into g.
// Mirrors the forward pass: decoder levels from the top down, then the encoder
// from the deepest level up.  A layer's gradient arrives masked by its ReLU,
// with the partial sums of its bias gradient taken (head_bwd, act_bwd*), which
// the last launch adds up.
int backward(lbpf_net* net, const float* dy)
{
    const int N = net->N, H = net->H, W = net->W, lv = net->levels;
    const long long P0 = (long long)N * H * W;
    cudaStream_t s = net->stream;
    float* g = net->g;
    auto bias = [&](int k) { return net->conv[k].part; };
    // weight gradient and data gradient (dx may be NULL) of conv k at level l
    // from the masked gradient dyk of its output
    auto cvb = [&](int k, const float* a, const float* b, int ca, int cb, const float* dyk, float* dx, int l) -> int {
        const Conv& c = net->conv[k];
        const int h = H >> l, w = W >> l;
        NK(conv3x3_wgrad_src(a, b, ca, cb, dyk, g + c.off_w, N, h, w, c.cout, s));
        if (dx) NK(conv3x3_fwd(dyk, c.wt, nullptr, dx, N, h, w, c.cout, c.cin, 0, s));
        return LBPF_OK;
    };
    int rc;
    int k = (int)net->conv.size();
    NK(head_bwd(net->top(), dy, net->p + net->off_hw, net->xin, kInPad, net->ga[0], net->head_part, P0, net->ch(0), s));
    for (int l = 0; l + 1 < lv; ++l) {  // decoder: the masked gradient of d[l] is in ga[l]
        k -= 2;
        const int c = net->ch(l), h = H >> l, w = W >> l;
        const long long Pl = P0 >> (2 * l);
        if ((rc = cvb(k + 1, net->da[l], nullptr, c, 0, net->ga[l], net->gb[l], l))) return rc;
        NK(act_bwd(net->da[l], net->gb[l], bias(k), Pl, c, s));
        // gradient of [up(below), e[l]] into ga[l]; its e[l] part stays there
        // until the encoder reads it
        if ((rc = cvb(k, net->below(l), net->e[l], net->ch(l + 1), c, net->gb[l], net->ga[l], l))) return rc;
        NK(act_bwd_up(net->below(l), net->ga[l], net->ga[l + 1], bias(l + 2 < lv ? k - 1 : 2 * lv - 1), N, h / 2, w / 2,
                      net->ch(l + 1), net->ch(l + 1) + c, s));
    }
    for (int l = lv - 1; l >= 0; --l) {  // encoder
        k -= 2;
        const int c = net->ch(l), h = H >> l, w = W >> l;
        const long long Pl = P0 >> (2 * l);
        float *a = net->ga[l], *b = net->gb[l];
        if (l + 1 < lv) {  // gradient of e[l]: pooled from level l + 1 (gb[l + 1]) plus the skip's (ga[l])
            NK(act_bwd_pool(net->e[l], net->gb[l + 1], net->ga[l], net->gb[l], bias(k + 1), N, h, w, c,
                            net->ch(l + 1) + c, net->ch(l + 1), s));
            std::swap(a, b);
        }
        // the masked gradient of e[l] is in a
        if ((rc = cvb(k + 1, net->ea[l], nullptr, c, 0, a, b, l))) return rc;
        NK(act_bwd(net->ea[l], b, bias(k), Pl, c, s));
        const int cin = net->conv[k].cin;
        if ((rc = cvb(k, l > 0 ? net->pl[l] : net->xin, nullptr, cin, 0, b, l > 0 ? a : nullptr, l))) return rc;
        if (l > 0 && a != net->gb[l]) std::swap(net->ga[l], net->gb[l]);  // level l - 1 reads gb[l]
    }
    NK(sum_partials(net->sums, s));
    return LBPF_OK;
}

}  // namespace

extern "C" int lbpf_net_forward(lbpf_net* net, const float* x, float* y)
{
    if (!net || !x) return LBPF_EINVAL;
    return forward(net, x, y);
}

extern "C" int lbpf_net_backward(lbpf_net* net, const float* dy)
{
    if (!net || !dy) return LBPF_EINVAL;
    NK(cudaMemsetAsync(net->g, 0, sizeof(float) * net->n_params, net->stream));
    return backward(net, dy);
}

extern "C" int lbpf_net_set_loss_weight(lbpf_net* net, float alpha)
{
    if (!net || !(alpha >= 0.f)) return LBPF_EINVAL;
    net->loss_alpha = alpha;
    return LBPF_OK;
}

extern "C" int lbpf_net_train_step(lbpf_net* net, const float* x, const float* target, float lr, double* loss)
{
    if (!net || !x || !target) return LBPF_EINVAL;
    int rc = forward(net, x, nullptr);
    if (rc) return rc;
    const long long n = (long long)net->N * net->H * net->W * kOut;
    NK(cudaMemsetAsync(net->d_loss, 0, sizeof(double), net->stream));
    NK(mse(net->out, target, x, kIn, kOut, net->loss_alpha, net->g_out, net->d_loss, n, net->stream));
    NK(cudaMemsetAsync(net->g, 0, sizeof(float) * net->n_params, net->stream));
    if ((rc = backward(net, net->g_out))) return rc;
    net->adam_t += 1;
    NK(adam(net->p, net->g, net->m, net->v, nullptr, net->n_params, lr, 0.9f, 0.999f, 1e-8f, net->adam_t, net->stream));
    if ((rc = refresh_bf16(net))) return rc;
    if (loss) {
        NK(cudaMemcpyAsync(loss, net->d_loss, sizeof(double), cudaMemcpyDeviceToHost, net->stream));
        NK(cudaStreamSynchronize(net->stream));
        if (conv_error() != 0) return net_fail(net, LBPF_ETIMEOUT, "a convolution block's bounded wait gave up");
    }
    return LBPF_OK;
}

extern "C" int lbpf_net_assemble(const float* phi, const float* u, const int* index, const float* crystal_tab,
                                 int n_crystals, float* x, long long sites, void* stream)
{
    if (!phi || !u || !x || sites < 1 || (n_crystals > 0 && !crystal_tab)) return LBPF_EINVAL;
    return assemble(phi, u, index, crystal_tab, n_crystals, x, sites, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? LBPF_OK
               : LBPF_ECUDA;
}

extern "C" int lbpf_net_apply(const float* y, float* phi, float* u, long long sites, void* stream)
{
    if (!y || !phi || !u || sites < 1) return LBPF_EINVAL;
    return apply(y, phi, u, sites, static_cast<cudaStream_t>(stream)) == cudaSuccess ? LBPF_OK : LBPF_ECUDA;
}

extern "C" int lbpf_net_delta(const float* phi0, const float* u0, const float* phi1, const float* u1, float* y,
                              long long sites, void* stream)
{
    if (!phi0 || !u0 || !phi1 || !u1 || !y || sites < 1) return LBPF_EINVAL;
    return delta(phi0, u0, phi1, u1, y, sites, static_cast<cudaStream_t>(stream)) == cudaSuccess ? LBPF_OK : LBPF_ECUDA;
}

extern "C" int lbpf_net_range_check(const float* phi, long long sites, float lo, float hi, unsigned int* count,
                                    void* stream)
{
    if (!phi || !count || sites < 1) return LBPF_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(count, 0, sizeof(unsigned int), s) != cudaSuccess) return LBPF_ECUDA;
    return range_count(phi, sites, lo, hi, count, s) == cudaSuccess ? LBPF_OK : LBPF_ECUDA;
}

extern "C" int lbpf_nn_conv3x3(const float* x, const void* wt, const float* bias, float* y, int n, int H, int W,
                               int cin, int cout, int relu, void* stream)
{
    const int n_tiles = (cout + 255) / 256;
    if (!x || !wt || !y || n < 1 || H < 1 || W < 1 || cin < 16 || cout < 16 || cin % 16 || cout % (16 * n_tiles))
        return LBPF_EINVAL;
    return conv3x3_fwd(x, static_cast<const __nv_bfloat16*>(wt), bias, y, n, H, W, cin, cout, relu,
                       static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? LBPF_OK
               : LBPF_ECUDA;
}

extern "C" int lbpf_nn_conv3x3_form(int H, int W, int cin, int cout, int* form)
{
    const int n_tiles = (cout + 255) / 256;
    if (!form || H < 1 || W < 1 || cin < 16 || cout < 16 || cin % 16 || cout % (16 * n_tiles)) return LBPF_EINVAL;
    *form = conv3x3_form(H, W, cin, cout);
    return LBPF_OK;
}

extern "C" int lbpf_nn_conv3x3_wgrad(const float* x, const float* dy, float* dwt, int n, int H, int W, int cin,
                                     int cout, void* stream)
{
    if (!x || !dy || !dwt || n < 1 || H < 1 || W < 1 || cin < 16 || cout < 16 || cin % 16 || cout % 16 ||
        (cin > 256 && cin % 32))
        return LBPF_EINVAL;
    return conv3x3_wgrad(x, dy, dwt, n, H, W, cin, cout, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? LBPF_OK
               : LBPF_ECUDA;
}

extern "C" int lbpf_nn_conv_error(int* word)
{
    if (!word) return LBPF_EINVAL;
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        return LBPF_ECUDA;
    }
    *word = conv_error();
    return *word < 0 ? LBPF_ECUDA : LBPF_OK;
}

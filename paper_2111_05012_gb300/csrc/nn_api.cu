// C ABI of the learned parallel-transport preconditioner: creation, weights,
// single-layer forward / backward (for parity tests), one Adam training step
// on a batch of (residual, error) pairs.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"

namespace {

amg_status nfail(amg_status st, const std::string& m) {
    amg_internal_set_error(m.c_str());
    return st;
}
#define NCK(x)                                                                                       \
    do {                                                                                             \
        cudaError_t e_ = (x);                                                                        \
        if (e_ != cudaSuccess) return nfail(AMG_ECUDA, std::string(#x) + " -> " + cudaGetErrorString(e_)); \
    } while (0)
#define NTRY(x)                       \
    do {                              \
        amg_status s_ = (x);          \
        if (s_ != AMG_OK) return s_;  \
    } while (0)

const int kRev[9] = {0, 5, 6, 7, 8, 1, 2, 3, 4};   // T_d^dag = T_{kRev[d]}

// float -> bfloat16 bits, round to nearest even
uint16_t to_bf16(float f) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    if ((u & 0x7f800000u) == 0x7f800000u) return (uint16_t)(u >> 16);   // inf / nan
    u += 0x7fffu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}
float from_bf16(uint16_t b) {
    uint32_t u = (uint32_t)b << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return f;
}

size_t layer_size(const amg_nn* nn, int l) { return (size_t)nn->ch[l + 1] * nn->ch[l] * 9 * 16 * 2; }

// upload bf16 weights and their adjoint: Wadj[b][a][d'] = W[a][b][rev d']^dag
amg_status upload_weights(amg_nn* nn) {
    for (int l = 0; l < nn->nlayers; ++l) {
        const int cin = nn->ch[l], cout = nn->ch[l + 1];
        const std::vector<float>& w = nn->w[l];
        std::vector<uint16_t> f(layer_size(nn, l)), a(layer_size(nn, l));
        for (size_t i = 0; i < f.size(); ++i) f[i] = to_bf16(w[i]);
        for (int oa = 0; oa < cout; ++oa)
            for (int ib = 0; ib < cin; ++ib)
                for (int d = 0; d < 9; ++d)
                    for (int s = 0; s < 4; ++s)
                        for (int t = 0; t < 4; ++t) {
                            // forward entry W[oa][ib][kRev[d]][t][s] -> adjoint entry Wadj[ib][oa][d][s][t], conjugated
                            size_t src = ((((size_t)oa * cin + ib) * 9 + kRev[d]) * 16 + t * 4 + s) * 2;
                            size_t dst = ((((size_t)ib * cout + oa) * 9 + d) * 16 + s * 4 + t) * 2;
                            a[dst] = f[src];
                            a[dst + 1] = to_bf16(-from_bf16(f[src + 1]));
                        }
        NCK(nn->wbf[l].ensure(f.size() * 2));
        NCK(nn->wadj[l].ensure(a.size() * 2));
        NCK(cudaMemcpy(nn->wbf[l].p, f.data(), f.size() * 2, cudaMemcpyHostToDevice));
        NCK(cudaMemcpy(nn->wadj[l].p, a.data(), a.size() * 2, cudaMemcpyHostToDevice));
    }
    return AMG_OK;
}

const GeomH& geom(amg_nn* nn) { return *amg_internal_geom(nn->d); }
size_t fbytes(amg_nn* nn) { return fine_spinor_bytes(1, geom(nn).V); }

// the layer's gradient on the device as host doubles (waits for the stream)
amg_status fetch_grad(amg_nn* nn, int l, double* out, cudaStream_t s) {
    NCK(cudaMemcpyAsync(out, nn->grad[l].p, layer_size(nn, l) * sizeof(double), cudaMemcpyDeviceToHost, s));
    NCK(cudaStreamSynchronize(s));
    return AMG_OK;
}

amg_status ensure_buffers(amg_nn* nn) {
    const size_t fb = fbytes(nn);
    int cmax = 1;
    for (int l = 0; l <= nn->nlayers; ++l) cmax = nn->ch[l] > cmax ? nn->ch[l] : cmax;
    for (int l = 0; l <= nn->nlayers; ++l) NCK(nn->act[l].ensure(fb * nn->ch[l]));
    NCK(nn->gbuf[0].ensure(fb * cmax));
    NCK(nn->gbuf[1].ensure(fb * cmax));
    NCK(nn->ework.ensure(fb));
    size_t pmax = 0;
    for (int l = 0; l < nn->nlayers; ++l) {
        pmax = std::max(pmax, ptconv_partials(nn->ch[l], nn->ch[l + 1]));
        NCK(nn->grad[l].ensure(layer_size(nn, l) * sizeof(double)));
    }
    NCK(nn->part.ensure(pmax * sizeof(double2)));
    return AMG_OK;
}

}  // namespace

amg_status nn_forward_internal(amg_nn* nn, const void* in32, void* out32, cudaStream_t s) {
    const void* cur = in32;
    for (int l = 0; l < nn->nlayers; ++l) {
        void* dst = (l == nn->nlayers - 1) ? out32 : nn->act[l + 1].p;
        NCK(launch_ptconv_forward(geom(nn), nn->ch[l], nn->ch[l + 1], amg_internal_links(nn->d, 1), nn->wbf[l].p,
                                  cur, dst, s));
        cur = dst;
    }
    return AMG_OK;
}

extern "C" {

amg_status amg_nn_create(amg_dirac* d, int nlayers, const int* channels, const float* weights, amg_nn** out) {
    if (!d || !channels || !weights || !out) return nfail(AMG_EINVAL, "amg_nn_create: NULL argument");
    if (nlayers < 1 || nlayers > AMG_NN_MAX_LAYERS) return nfail(AMG_EINVAL, "amg_nn_create: 1..4 layers");
    if (channels[0] != 1 || channels[nlayers] != 1)
        return nfail(AMG_EINVAL, "amg_nn_create: the network maps one field to one field");
    for (int l = 0; l <= nlayers; ++l)
        if (channels[l] < 1 || channels[l] > 4) return nfail(AMG_EINVAL, "amg_nn_create: 1..4 channels per layer");
    amg_nn* nn = new amg_nn();
    nn->d = d;
    nn->nlayers = nlayers;
    for (int l = 0; l <= nlayers; ++l) nn->ch[l] = channels[l];
    const float* p = weights;
    for (int l = 0; l < nlayers; ++l) {
        size_t n = layer_size(nn, l);
        nn->w.emplace_back(p, p + n);
        nn->m.emplace_back(n, 0.0);
        nn->v.emplace_back(n, 0.0);
        p += n;
    }
    amg_status st = upload_weights(nn);
    if (st == AMG_OK) st = ensure_buffers(nn);
    if (st != AMG_OK) {
        delete nn;
        return st;
    }
    *out = nn;
    return AMG_OK;
}

void amg_nn_destroy(amg_nn* nn) { delete nn; }

amg_status amg_nn_get_weights(amg_nn* nn, int effective, float* host_out) {
    if (!nn || !host_out) return nfail(AMG_EINVAL, "amg_nn_get_weights: NULL argument");
    float* p = host_out;
    for (int l = 0; l < nn->nlayers; ++l) {
        for (size_t i = 0; i < nn->w[l].size(); ++i) p[i] = effective ? from_bf16(to_bf16(nn->w[l][i])) : nn->w[l][i];
        p += nn->w[l].size();
    }
    return AMG_OK;
}

amg_status amg_nn_layer_forward(amg_nn* nn, int layer, const float* in, float* out, amg_stream stream) {
    if (!nn || !in || !out || layer < 0 || layer >= nn->nlayers) return nfail(AMG_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    const GeomH& g = geom(nn);
    const int cin = nn->ch[layer], cout = nn->ch[layer + 1];
    NCK(launch_pack_spinor(1, g, in, nn->gbuf[0].p, cin, s));
    NCK(launch_ptconv_forward(g, cin, cout, amg_internal_links(nn->d, 1), nn->wbf[layer].p, nn->gbuf[0].p,
                              nn->gbuf[1].p, s));
    NCK(launch_unpack_spinor(1, g, nn->gbuf[1].p, out, cout, s));
    return AMG_OK;
}

amg_status amg_nn_layer_backward(amg_nn* nn, int layer, const float* in, const float* grad_out, float* grad_in,
                                 double* grad_w, amg_stream stream) {
    if (!nn || !in || !grad_out || layer < 0 || layer >= nn->nlayers) return nfail(AMG_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    const GeomH& g = geom(nn);
    const int cin = nn->ch[layer], cout = nn->ch[layer + 1];
    NCK(launch_pack_spinor(1, g, in, nn->gbuf[0].p, cin, s));
    NCK(launch_pack_spinor(1, g, grad_out, nn->gbuf[1].p, cout, s));
    if (grad_w) {
        NCK(launch_ptconv_wgrad(g, cin, cout, amg_internal_links(nn->d, 1), nn->gbuf[0].p, nn->gbuf[1].p,
                                nn->part.as<double2>(), nullptr, false, nn->grad[layer].as<double2>(), s));
        NTRY(fetch_grad(nn, layer, grad_w, s));
    }
    if (grad_in) {
        NCK(launch_ptconv_forward(g, cout, cin, amg_internal_links(nn->d, 1), nn->wadj[layer].p, nn->gbuf[1].p,
                                  nn->gbuf[0].p, s));
        NCK(launch_unpack_spinor(1, g, nn->gbuf[0].p, grad_in, cin, s));
    }
    NCK(cudaStreamSynchronize(s));
    return AMG_OK;
}

amg_status amg_nn_apply(amg_nn* nn, const float* in, float* out, amg_stream stream) {
    if (!nn || !in || !out) return nfail(AMG_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    const GeomH& g = geom(nn);
    NCK(launch_pack_spinor(1, g, in, nn->act[0].p, 1, s));
    NTRY(nn_forward_internal(nn, nn->act[0].p, nn->ework.p, s));
    NCK(launch_unpack_spinor(1, g, nn->ework.p, out, 1, s));
    return AMG_OK;
}

amg_status amg_nn_train_step(amg_nn* nn, const float* r, const float* e, int npairs, double lr, double* loss_out,
                             amg_stream stream) {
    if (!nn || !r || !e || npairs < 1 || !(lr > 0)) return nfail(AMG_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    const GeomH& g = geom(nn);
    const int L = nn->nlayers;
    NCK(nn->norms.ensure(npairs * sizeof(double2)));
    // every pair's gradient is summed on the device, scaled by 1 / |e|^2 as it is added; the
    // host waits once for the whole batch
    for (int p = 0; p < npairs; ++p) {
        double2* norm = nn->norms.as<double2>() + p;
        const float* target = e + (size_t)p * g.V * 24;
        if (((uintptr_t)target & 15) != 0) {
            // the loss reads its target in 16-byte words: an unaligned one is copied, pair by pair
            NCK(cudaMemcpyAsync(nn->ework.p, target, (size_t)g.V * 24 * sizeof(float), cudaMemcpyDeviceToDevice, s));
            target = nn->ework.as<float>();
        }
        NCK(launch_pack_spinor(1, g, r + (size_t)p * g.V * 24, nn->act[0].p, 1, s));
        for (int l = 0; l < L; ++l)
            NCK(launch_ptconv_forward(g, nn->ch[l], nn->ch[l + 1], amg_internal_links(nn->d, 1), nn->wbf[l].p,
                                      nn->act[l].p, nn->act[l + 1].p, s, l == L - 1 ? target : nullptr,
                                      nn->part.as<double2>(), norm));
        const void* gout = nn->act[L].p;   // y - e
        int gi = 0;
        for (int l = L - 1; l >= 0; --l) {
            NCK(launch_ptconv_wgrad(g, nn->ch[l], nn->ch[l + 1], amg_internal_links(nn->d, 1), nn->act[l].p, gout,
                                    nn->part.as<double2>(), norm, p > 0, nn->grad[l].as<double2>(), s));
            if (l > 0) {
                NCK(launch_ptconv_forward(g, nn->ch[l + 1], nn->ch[l], amg_internal_links(nn->d, 1), nn->wadj[l].p,
                                          gout, nn->gbuf[gi].p, s));
                gout = nn->gbuf[gi].p;
                gi ^= 1;
            }
        }
    }
    std::vector<std::vector<double>> gsum(L);
    for (int l = 0; l < L; ++l) gsum[l].resize(layer_size(nn, l));
    std::vector<double2> norms(npairs);
    NCK(cudaMemcpyAsync(norms.data(), nn->norms.p, npairs * sizeof(double2), cudaMemcpyDeviceToHost, s));
    for (int l = 0; l < L; ++l) NTRY(fetch_grad(nn, l, gsum[l].data(), s));
    double loss = 0;
    for (const double2& v : norms) {
        if (!(v.y > 0)) return nfail(AMG_EINVAL, "amg_nn_train_step: zero error vector");
        loss += v.x / v.y;
        if (!std::isfinite(loss)) return nfail(AMG_NAN, "amg_nn_train_step: non-finite loss");
    }
    // Adam on the real and imaginary parts; d/d(Re W) = 2 Re G, d/d(Im W) = 2 Im G (mean over pairs)
    const double b1 = 0.9, b2 = 0.999, eps = 1e-8;
    nn->adam_t++;
    const double c1 = 1.0 - std::pow(b1, nn->adam_t), c2 = 1.0 - std::pow(b2, nn->adam_t);
    for (int l = 0; l < L; ++l)
        for (size_t i = 0; i < nn->w[l].size(); ++i) {
            const double gr = 2.0 * gsum[l][i] / npairs;
            nn->m[l][i] = b1 * nn->m[l][i] + (1 - b1) * gr;
            nn->v[l][i] = b2 * nn->v[l][i] + (1 - b2) * gr * gr;
            const double mh = nn->m[l][i] / c1, vh = nn->v[l][i] / c2;
            nn->w[l][i] = (float)(nn->w[l][i] - lr * mh / (std::sqrt(vh) + eps));
        }
    NTRY(upload_weights(nn));
    if (loss_out) *loss_out = loss / npairs;
    return AMG_OK;
}

void amg_train_params_default(amg_train_params* p) {
    if (!p) return;
    p->npairs = 4096;
    p->batch = 16;
    p->lr = 1e-3;
    p->seed = 5;
}

amg_status amg_learned_train(amg_hierarchy* h, amg_nn* nn, const amg_train_params* p, double* losses,
                             amg_stream stream) {
    if (!h || !nn || !p || p->npairs < 1 || p->batch < 1 || !(p->lr > 0))
        return nfail(AMG_EINVAL, "amg_learned_train: bad argument");
    amg_dirac* d = amg_internal_hierarchy_dirac(h);
    if (d != nn->d) return nfail(AMG_EINVAL, "amg_learned_train: network and hierarchy use different operators");
    cudaStream_t s = (cudaStream_t)stream;
    const GeomH& g = geom(nn);
    const size_t n = (size_t)g.V * 12;   // complex numbers per field
    const size_t f64 = n * 16, f32 = n * 8;
    DevBuf e0, w, e1, r1, rb, eb;
    NCK(e0.ensure(f64));
    NCK(w.ensure(f64));
    NCK(e1.ensure(f64));
    NCK(r1.ensure(f64));
    NCK(rb.ensure(f32 * p->batch));
    NCK(eb.ensure(f32 * p->batch));
    const int steps = p->npairs / p->batch;
    if (steps < 1) return nfail(AMG_EINVAL, "amg_learned_train: npairs < batch");
    for (int st = 0; st < steps; ++st) {
        for (int q = 0; q < p->batch; ++q) {
            const uint64_t k = (uint64_t)st * p->batch + q;
            // e0: Gaussian field k of stream (seed, AMG_RNG_STREAM_NN); e = e0 - M D e0, r = D e
            NCK(launch_random_normal(p->seed, AMG_RNG_STREAM_NN, k * n, n, e0.as<double>(), s));
            NTRY(amg_apply_D(d, e0.p, w.p, 1, AMG_F64, stream));
            NTRY(amg_precondition(h, w.as<double>(), e1.as<double>(), stream));
            NCK(launch_axpby(0, make_double2(1, 0), e0.p, make_double2(-1, 0), e1.p, n, s));
            NTRY(amg_apply_D(d, e1.p, r1.p, 1, AMG_F64, stream));
            NCK(launch_convert_flat(0, 1, e1.p, (char*)eb.p + q * f32, n, s));
            NCK(launch_convert_flat(0, 1, r1.p, (char*)rb.p + q * f32, n, s));
        }
        double loss = 0;
        NTRY(amg_nn_train_step(nn, rb.as<float>(), eb.as<float>(), p->batch, p->lr, &loss, stream));
        if (losses) losses[st] = loss;
    }
    NCK(cudaStreamSynchronize(s));
    return AMG_OK;
}

}  // extern "C"

// Host-side internals shared by the C-ABI translation units.
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "kernels.h"
#include "lqcd_amg.h"

// Owning device buffer that only grows.
struct DevBuf {
    void* p = nullptr;
    size_t n = 0;
    DevBuf() = default;
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
    DevBuf(DevBuf&& o) noexcept : p(o.p), n(o.n) {
        o.p = nullptr;
        o.n = 0;
    }
    ~DevBuf() {
        if (p) cudaFree(p);
    }
    cudaError_t ensure(size_t bytes) {
        if (bytes <= n) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
        cudaError_t e = cudaMalloc(&p, bytes ? bytes : 16);
        if (e == cudaSuccess) n = bytes;
        return e;
    }
    template <typename T> T* as() const { return (T*)p; }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
    void swap(DevBuf& o) noexcept {
        void* tp = p;
        p = o.p;
        o.p = tp;
        size_t tn = n;
        n = o.n;
        o.n = tn;
    }
};

#define AMG_NN_MAX_LAYERS 4

// Learned parallel-transport preconditioner (layers of ptconv.cu).
struct amg_nn {
    amg_dirac* d = nullptr;
    int nlayers = 0;
    int ch[AMG_NN_MAX_LAYERS + 1] = {0};
    std::vector<std::vector<float>> w;      // FP32 master weights [cout][cin][9][4][4][re,im]
    std::vector<std::vector<double>> m, v;  // Adam moments
    int adam_t = 0;
    DevBuf wbf[AMG_NN_MAX_LAYERS];          // bfloat16 weights of the forward layers
    DevBuf wadj[AMG_NN_MAX_LAYERS];         // bfloat16 adjoint weights (input gradient)
    DevBuf act[AMG_NN_MAX_LAYERS + 1];      // activations, FP32 internal fields x channels
    DevBuf gbuf[2];                         // gradient fields
    DevBuf ework;                           // output field; in a training step an unaligned pair's target
    DevBuf part;                            // reduction partials
    DevBuf grad[AMG_NN_MAX_LAYERS];         // weight gradients, summed over a batch's pairs
    DevBuf norms;                           // per pair (|y - e|^2, |e|^2)
};

// accessors implemented in api.cu
const GeomH* amg_internal_geom(const amg_dirac* d);
amg_dirac* amg_internal_hierarchy_dirac(amg_hierarchy* h);
const void* amg_internal_links(const amg_dirac* d, int prec);
void amg_internal_set_error(const char* msg);

// PT-conv launchers (ptconv.cu)
size_t ptconv_partials(int cin, int cout);   // double2 entries of part for a layer
// out = layer(in).  With target (one output channel, canonical floats): out = layer(in) - target,
// and *norms = (|out|^2, |target|^2), through the CTAs' shares in part.
cudaError_t launch_ptconv_forward(const GeomH& g, int cin, int cout, const void* U32, const void* Wbf16,
                                  const void* in, void* out, cudaStream_t s, const float* target = nullptr,
                                  double2* part = nullptr, double2* norms = nullptr);
// G (+)= the layer's weight gradient [cout][cin][9][4][4] (device), over norm->y if norm is given
cudaError_t launch_ptconv_wgrad(const GeomH& g, int cin, int cout, const void* U32, const void* in, const void* gout,
                                double2* part, const double2* norm, bool add, double2* G, cudaStream_t s);

// network forward on FP32 internal fields: out = N(in) (nn_api.cu)
amg_status nn_forward_internal(amg_nn* nn, const void* in32, void* out32, cudaStream_t s);

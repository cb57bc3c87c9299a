// Transfer between the fine lattice and the first coarse lattice (Sec. 3):
// restriction x(I) = <I|x> (Eq. 5), prolongation |x'> = sum_I x(I)|I> (Eq. 6),
// the block orthonormalisation <I|J> = delta_IJ and the Galerkin coarse
// operator D_c(I, J) = <I|D|J> (Eq. 7).  |X, s, i> is test vector i projected
// to chirality s (spins 0,1 or 2,3) and restricted to block X; coarse dof
// index I = s * nvec + i.  One CTA works on one block, one thread per site.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace {

Geom make_geom(const GeomH& h) {
    Geom g;
    for (int i = 0; i < 4; ++i) g.L[i] = h.L[i];
    g.stride[0] = 1;
    g.stride[1] = h.L[0];
    g.stride[2] = h.L[0] * h.L[1];
    g.stride[3] = h.L[0] * h.L[1] * h.L[2];
    g.V = h.V;
    g.antiperiodic = h.antiperiodic;
    return g;
}
Blocking make_blocking(const GeomH& g, const BlockH& b) {
    Blocking k;
    k.Vb = 1;
    k.Vc = 1;
    for (int i = 0; i < 4; ++i) {
        k.b[i] = b.b[i];
        k.C[i] = g.L[i] / b.b[i];
        k.Vb *= k.b[i];
        k.Vc *= k.C[i];
    }
    return k;
}

template <typename TC> struct CStore;
template <> struct CStore<double> {
    DEV static void st(void* p, size_t i, cx<double> v) { ((double2*)p)[i] = make_double2(v.re, v.im); }
    DEV static cx<double> ld(const void* p, size_t i) {
        double2 t = ((const double2*)p)[i];
        return {t.x, t.y};
    }
};
template <> struct CStore<float> {
    DEV static void st(void* p, size_t i, cx<float> v) { ((float2*)p)[i] = make_float2(v.re, v.im); }
    DEV static cx<float> ld(const void* p, size_t i) {
        float2 t = ((const float2*)p)[i];
        return {t.x, t.y};
    }
};

// ------------------------------------------------------------ raw vector loads
// A test vector at one site as loaded from memory, unpacked only when used, so
// that the loads of several vectors can be in flight together without holding
// all of them unpacked in registers.
template <class PV> struct RawSite;
template <> struct RawSite<P64> {
    double2 r[12];
    DEV void load(const void* base, int V, int s) {
#pragma unroll
        for (int k = 0; k < 12; ++k) r[k] = __ldg((const double2*)base + (size_t)k * V + s);
    }
    DEV cx<double> get(int k) const { return {r[k].x, r[k].y}; }
};
template <> struct RawSite<P32> {
    float4 r[6];
    DEV void load(const void* base, int V, int s) {
#pragma unroll
        for (int c = 0; c < 6; ++c) r[c] = __ldg((const float4*)base + (size_t)c * V + s);
    }
    DEV cx<float> get(int k) const {
        const float4 t = r[k >> 1];
        return (k & 1) ? cx<float>{t.z, t.w} : cx<float>{t.x, t.y};
    }
};
template <> struct RawSite<P16> {   // three uint4 of halves, then the per-site scale (SpinorIO<P16> layout)
    uint4 r[3];
    float sc;
    DEV void load(const void* base, int V, int s) {
        const uint4* p = (const uint4*)base;
#pragma unroll
        for (int c = 0; c < 3; ++c) r[c] = __ldg(p + (size_t)c * V + s);
        sc = __ldg((const float*)(p + (size_t)3 * V) + s);
    }
    DEV cx<float> get(int k) const {
        const uint4 t = r[k >> 2];
        const unsigned w = (k & 3) == 0 ? t.x : (k & 3) == 1 ? t.y : (k & 3) == 2 ? t.z : t.w;
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
        return {f.x * sc, f.y * sc};
    }
};
// vectors whose loads a thread keeps in flight together
template <class PV> constexpr int kVecGroup = PV::id == 2 ? 4 : 2;

// A fine vector as the caller holds it: 24 floats per site, one site after another (aligned to 16
// bytes); blocks have runs of sites along x, so a warp's six loads use whole sectors.
struct CanonF32 {
    DEV static void load(const void* base, int, int s, cx<float> v[12]) {
        const float4* p = (const float4*)base + (size_t)s * 6;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const float4 t = __ldg(p + c);
            v[2 * c] = {t.x, t.y};
            v[2 * c + 1] = {t.z, t.w};
        }
    }
    DEV static void store(void* base, int, int s, const cx<float> v[12]) {
        float4* p = (float4*)base + (size_t)s * 6;
#pragma unroll
        for (int c = 0; c < 6; ++c) p[c] = make_float4(v[2 * c].re, v[2 * c].im, v[2 * c + 1].re, v[2 * c + 1].im);
    }
};

// ------------------------------------------------------------ restriction
// One CTA per block and group of NB right-hand sides, one thread per site: the site's share of
// <X,s,i|psi_r> for a group of test vectors (their loads in flight together, the next group's
// under the products of this one in a batch), summed over the warp by transposed shuffles and over the warps
// in shared memory.  The test vectors are most of the traffic (96 or 52 bytes per site and vector
// against 96 per right-hand side), so a batch reads them once per NB = 4 vectors; every
// right-hand side goes through the same sums whatever NB is.  Bound by HBM: FP32 vectors,
// 24^3 x 48, 24 of them, four right-hand sides 554 -> 339 us (1.78 GB, 262 us at the copy rate).
// IO: the layout of the fine vectors (internal, or the caller's).
template <class PV, int NB> constexpr int kGroupOf = NB == 4 ? 2 : kVecGroup<PV>;
template <class PF, class PV, typename TC, int NB = 1, class IO = SpinorIO<PF>>
DEV void restrict_body(const Geom& g, const Blocking& bk, int nvec, const void* __restrict__ vecs,
                       const void* __restrict__ fine, size_t fstride, void* coarse, int nr, int by, int gy) {
    using T = typename PF::T;
    constexpr int G = kGroupOf<PV, NB>, NQ = 4 * G * NB;   // per vector and right-hand side: d0.re, d0.im, d1.re, d1.im
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T>* part = reinterpret_cast<cx<T>*>(smem_raw);   // [nwarps][NB][2*nvec]
    T* partf = reinterpret_cast<T*>(smem_raw);
    const int nc = 2 * nvec;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t vb = spinor_bytes<PV>(g.V);
    const int qi = transposed_index<NQ>(lane);
    const bool writer = (lane & (32 / NQ - 1)) == 0;
    // the loads of the group of vectors from i0 on
    auto fetch = [&](RawSite<PV> (&raw)[G], int i0, int s) {
#pragma unroll
        for (int u = 0; u < G; ++u)
            if (i0 + u < nvec) raw[u].load((const char*)vecs + (size_t)(i0 + u) * vb, g.V, s);
    };
    for (int Xi = by; Xi < bk.Vc; Xi += gy) {
        const int l = threadIdx.x;
        const bool active = l < bk.Vb;
        int c[4], s = 0;
        cx<T> psi[NB][12];
        RawSite<PV> raw[G];
        if (active) {
            s = block_site(g, bk, Xi, l, c);
            if (NB > 1) fetch(raw, 0, s);
#pragma unroll
            for (int r = 0; r < NB; ++r) {
                if (r < nr) IO::load((const char*)fine + r * fstride, g.V, s, psi[r]);
                else
#pragma unroll
                    for (int k = 0; k < 12; ++k) psi[r][k] = czero<T>();
            }
        }
        for (int i0 = 0; i0 < nvec; i0 += G) {
            if (NB == 1 && active) fetch(raw, i0, s);
            T q[NQ];
#pragma unroll
            for (int u = 0; u < G; ++u) {
                const RawSite<PV> v = raw[u];
                if (NB > 1 && active && i0 + G + u < nvec)
                    raw[u].load((const char*)vecs + (size_t)(i0 + G + u) * vb, g.V, s);
#pragma unroll
                for (int r = 0; r < NB; ++r) {
                    cx<T> d0 = czero<T>(), d1 = czero<T>();
                    if (active && i0 + u < nvec) {
#pragma unroll
                        for (int k = 0; k < 6; ++k) {
                            cfmac(d0, ccast<T>(v.get(k)), psi[r][k]);
                            cfmac(d1, ccast<T>(v.get(6 + k)), psi[r][6 + k]);
                        }
                    }
                    T* o = q + 4 * (u * NB + r);
                    o[0] = d0.re;
                    o[1] = d0.im;
                    o[2] = d1.re;
                    o[3] = d1.im;
                }
            }
            const T tot = transposed_warp_sum<NQ>(q, lane);
            const int r = (qi >> 2) % NB, comp = qi & 3, i = i0 + (qi >> 2) / NB;
            if (writer && i < nvec)
                partf[2 * ((warp * NB + r) * nc + (comp < 2 ? i : nvec + i)) + (comp & 1)] = tot;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < nr * nc; j += blockDim.x) {
            const int r = j / nc, q = j - r * nc;
            cx<T> t = czero<T>();
            for (int w = 0; w < nw; ++w) t = t + part[(w * NB + r) * nc + q];
            CStore<TC>::st(coarse, ((size_t)r * bk.Vc + Xi) * nc + q, ccast<TC>(t));
        }
        __syncthreads();
    }
}

// group of right-hand sides = blockIdx.x (the fast grid index): the CTAs of one block for all
// groups of a batch are launched together and read the same test-vector lines at about the same
// time, so L2 serves the repeats and DRAM sees each line about once
template <class PF, class PV, typename TC, int NB, class IO>
__global__ void __launch_bounds__(256, 1)
    restrict_batch_kernel(Geom g, Blocking bk, int nvec, const void* __restrict__ vecs, const void* __restrict__ fine,
                    size_t fstride, void* coarse, int nrhs, int per) {
    const int r0 = blockIdx.x * per;
    restrict_body<PF, PV, TC, NB, IO>(g, bk, nvec, vecs, (const char*)fine + r0 * fstride, fstride,
                                      (char*)coarse + r0 * (size_t)bk.Vc * 2 * nvec * sizeof(cx<TC>),
                                      min(per, nrhs - r0), blockIdx.y, gridDim.y);
}
// one right-hand side per CTA
template <class PF, class PV, typename TC, class IO>
__global__ void restrict_kernel(Geom g, Blocking bk, int nvec, const void* __restrict__ vecs,
                                const void* __restrict__ fine, size_t fstride, void* coarse) {
    restrict_body<PF, PV, TC, 1, IO>(g, bk, nvec, vecs, (const char*)fine + blockIdx.x * fstride, fstride,
                                     (char*)coarse + blockIdx.x * (size_t)bk.Vc * 2 * nvec * sizeof(cx<TC>), 1,
                                     blockIdx.y, gridDim.y);
}
// ragged batch: bc = R f32 for every problem in one launch (one CTA per block)
template <class PV>
__global__ void restrict_ragged_kernel(const RaggedDev* __restrict__ d, const int* __restrict__ off, int np) {
    int p, bx, gx;
    ragged_locate(off, np, p, bx, gx);
    const RaggedDev& q = d[p];
    restrict_body<P32, PV, float>(q.g, q.bk, q.nvec, q.vecs, q.f32, 0, q.bc, 1, bx, gx);
}

// ------------------------------------------------------------ prolongation
// One CTA per block and group of NB right-hand sides, one thread per site:
// psi_r'(x) = sum_{s,i} x_c(X, s, i) P_s v_i(x), the loads of a group of test vectors in flight
// under the products of the group before in a batch.  24^3 x 48, 24 FP32 vectors, four right-hand sides:
// 485 -> 344 us.
template <class PF, class PV, typename TC, int NB = 1, class IO = SpinorIO<PF>>
DEV void prolong_body(const Geom& g, const Blocking& bk, int nvec, const void* __restrict__ vecs,
                      const void* __restrict__ coarse, void* fine, size_t fstride, int nr, int by, int gy) {
    using T = typename PF::T;
    constexpr int G = kGroupOf<PV, NB>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<T>* xc = reinterpret_cast<cx<T>*>(smem_raw);   // [2*nvec][NB]
    const int nc = 2 * nvec;
    const size_t vb = spinor_bytes<PV>(g.V);
    // the loads of the group of vectors from i0 on
    auto fetch = [&](RawSite<PV> (&raw)[G], int i0, int s) {
#pragma unroll
        for (int u = 0; u < G; ++u)
            if (i0 + u < nvec) raw[u].load((const char*)vecs + (size_t)(i0 + u) * vb, g.V, s);
    };
    for (int Xi = by; Xi < bk.Vc; Xi += gy) {
        const int l = threadIdx.x;
        const bool active = l < bk.Vb;
        int c[4], s = 0;
        RawSite<PV> raw[G];
        if (active) {
            s = block_site(g, bk, Xi, l, c);
            if (NB > 1) fetch(raw, 0, s);
        }
        for (int j = threadIdx.x; j < NB * nc; j += blockDim.x) {
            const int r = j / nc, q = j - r * nc;
            xc[q * NB + r] = r < nr ? ccast<T>(CStore<TC>::ld(coarse, ((size_t)r * bk.Vc + Xi) * nc + q)) : czero<T>();
        }
        __syncthreads();
        if (active) {
            cx<T> out[NB][12];
#pragma unroll
            for (int r = 0; r < NB; ++r)
#pragma unroll
                for (int k = 0; k < 12; ++k) out[r][k] = czero<T>();
            for (int i0 = 0; i0 < nvec; i0 += G) {
                if (NB == 1) fetch(raw, i0, s);
#pragma unroll
                for (int u = 0; u < G; ++u) {
                    const RawSite<PV> v = raw[u];
                    if (NB > 1 && i0 + G + u < nvec) raw[u].load((const char*)vecs + (size_t)(i0 + G + u) * vb, g.V, s);
                    if (i0 + u < nvec) {
#pragma unroll
                        for (int r = 0; r < NB; ++r) {
                            const cx<T> a0 = xc[(i0 + u) * NB + r], a1 = xc[(nvec + i0 + u) * NB + r];
#pragma unroll
                            for (int k = 0; k < 6; ++k) {
                                cfma(out[r][k], a0, ccast<T>(v.get(k)));
                                cfma(out[r][6 + k], a1, ccast<T>(v.get(6 + k)));
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < NB; ++r)
                if (r < nr) IO::store((char*)fine + r * fstride, g.V, s, out[r]);
        }
        __syncthreads();
    }
}

// group of right-hand sides = blockIdx.x, as in restrict_kernel
template <class PF, class PV, typename TC, int NB, class IO>
__global__ void __launch_bounds__(256, 1)
    prolong_batch_kernel(Geom g, Blocking bk, int nvec, const void* __restrict__ vecs, const void* __restrict__ coarse,
                   void* fine, size_t fstride, int nrhs, int per) {
    const int r0 = blockIdx.x * per;
    prolong_body<PF, PV, TC, NB, IO>(g, bk, nvec, vecs,
                                     (const char*)coarse + r0 * (size_t)bk.Vc * 2 * nvec * sizeof(cx<TC>),
                                     (char*)fine + r0 * fstride, fstride, min(per, nrhs - r0), blockIdx.y, gridDim.y);
}
// one right-hand side per CTA
template <class PF, class PV, typename TC, class IO>
__global__ void prolong_kernel(Geom g, Blocking bk, int nvec, const void* __restrict__ vecs,
                               const void* __restrict__ coarse, void* fine, size_t fstride) {
    prolong_body<PF, PV, TC, 1, IO>(g, bk, nvec, vecs,
                                    (const char*)coarse + blockIdx.x * (size_t)bk.Vc * 2 * nvec * sizeof(cx<TC>),
                                    (char*)fine + blockIdx.x * fstride, fstride, 1, blockIdx.y, gridDim.y);
}
// ragged batch: z = P xc for every problem in one launch (one CTA per block)
template <class PV>
__global__ void prolong_ragged_kernel(const RaggedDev* __restrict__ d, const int* __restrict__ off, int np) {
    int p, bx, gx;
    ragged_locate(off, np, p, bx, gx);
    const RaggedDev& q = d[p];
    prolong_body<P32, PV, float>(q.g, q.bk, q.nvec, q.vecs, q.xc, q.z, 0, 1, bx, gx);
}

// ------------------------------------------------------------ orthonormalisation
// Per (block, chirality): Gram-Schmidt over i = 0..nvec-1 in index order against
// the previous (orthonormal) vectors, in FP64.  Each projection takes the
// coefficients <v_j, w> of all previous vectors in one pass (classical form:
// per-warp sums into shared memory, one barrier, one cross-warp sum per
// coefficient), then subtracts them in a second pass over the vectors.  A second
// projection follows only if the first removed more than three quarters of
// |w|^2: against an orthonormal set one projection leaves w orthogonal to about
// eps |w0| / |w| <= 2 eps otherwise (the DGKS test).  Either way the result is
// the QR factor with a positive diagonal to rounding, the vectors that
// projecting one vector after another gives.  orthonormalise_kernel does this
// for FP64 vectors, orthonormalise_pairs_kernel for FP32 vectors.

// chirality half chi of a fine field at one site (plain loads: written earlier in the launch)
template <class PV> DEV void load_chirality(const void* base, int V, int s, int chi, cx<typename PV::T> v[6]);
template <> DEV void load_chirality<P32>(const void* base, int V, int s, int chi, cx<float> v[6]) {
    const float4* p = (const float4*)base + (size_t)3 * chi * V;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float4 t = p[(size_t)c * V + s];
        v[2 * c] = {t.x, t.y};
        v[2 * c + 1] = {t.z, t.w};
    }
}
template <> DEV void load_chirality<P64>(const void* base, int V, int s, int chi, cx<double> v[6]) {
    const double2* p = (const double2*)base + (size_t)6 * chi * V;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double2 t = p[(size_t)k * V + s];
        v[k] = {t.x, t.y};
    }
}
__global__ void __launch_bounds__(512) orthonormalise_kernel(Geom g, Blocking bk, int nvec, void* vecs, int* err) {
    __shared__ double red[3 * 32];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<double>* part = reinterpret_cast<cx<double>*>(smem_raw);   // [nwarps][nvec]
    cx<double>* coef = part + (size_t)(blockDim.x / 32) * nvec;    // [nvec]
    const int Xi = blockIdx.x, chi = blockIdx.y;
    const int l = threadIdx.x, lane = l & 31, warp = l >> 5, nw = blockDim.x >> 5;
    const bool active = l < bk.Vb;
    const size_t vb = spinor_bytes<P64>(g.V);
    int c[4], s = 0;
    if (active) s = block_site(g, bk, Xi, l, c);
    auto load_half = [&](int j, cx<double> (&q)[6]) {
        if (active) {
            cx<double> u[6];
            load_chirality<P64>((const char*)vecs + j * vb, g.V, s, chi, u);
#pragma unroll
            for (int k = 0; k < 6; ++k) q[k] = u[k];
        } else {
#pragma unroll
            for (int k = 0; k < 6; ++k) q[k] = czero<double>();
        }
    };
    for (int i = 0; i < nvec; ++i) {
        cx<double> w[6];
        load_half(i, w);
        double n0[1] = {0};
        for (int k = 0; k < 6; ++k) n0[0] += norm2(w[k]);
        block_sum<double, 1>(n0, red);
        for (int pass = 0; pass < 2 && i > 0; ++pass) {
            if (pass == 1) {   // a second projection only after a large cancellation
                double n1[1] = {0};
                for (int k = 0; k < 6; ++k) n1[0] += norm2(w[k]);
                block_sum<double, 1>(n1, red);
                if (n1[0] > 0.25 * n0[0]) break;
            }
            for (int j = 0; j < i; ++j) {
                cx<double> d = czero<double>();
                if (active) {
                    cx<double> u[6];
                    load_chirality<P64>((const char*)vecs + j * vb, g.V, s, chi, u);
#pragma unroll
                    for (int k = 0; k < 6; ++k) cfmac(d, u[k], w[k]);
                }
                // the upper half of the warp ends with the sum of the imaginary parts
                double q[2] = {d.re, d.im};
                const double tot = transposed_warp_sum<2>(q, lane);
                if ((lane & 15) == 0) reinterpret_cast<double*>(part + warp * nvec + j)[lane >> 4] = tot;
            }
            __syncthreads();
            for (int j = l; j < i; j += blockDim.x) {
                cx<double> t = czero<double>();
                for (int ww = 0; ww < nw; ++ww) t = t + part[ww * nvec + j];
                coef[j] = t;
            }
            __syncthreads();
            for (int j = 0; j < i && active; ++j) {
                cx<double> u[6];
                load_chirality<P64>((const char*)vecs + j * vb, g.V, s, chi, u);
                const cx<double> cc = -coef[j];
#pragma unroll
                for (int k = 0; k < 6; ++k) cfma(w[k], cc, u[k]);
            }
            __syncthreads();   // part / coef are rewritten by the next pass
        }
        double nn[1] = {0};
        for (int k = 0; k < 6; ++k) nn[0] += norm2(w[k]);
        block_sum<double, 1>(nn, red);
        // rank test: |w| <= 1e-12 |w0|
        const double rtol2 = 1e-24;
        if (!(nn[0] > rtol2 * n0[0])) {
            if (threadIdx.x == 0) atomicExch(err, 1);
            nn[0] = 1.0;
        }
        double inv = 1.0 / sqrt(nn[0]);
        if (active) {
            // the other chirality half belongs to the CTA (Xi, 1 - chi): write ours only
            cx<double> hv[6];
            for (int k = 0; k < 6; ++k) hv[k] = ccast<double>(inv * w[k]);
            SpinorIO<P64>::store_half((char*)vecs + i * vb, g.V, s, chi, hv);
        }
        __syncthreads();
    }
}

// ---- FP32 vectors: the same Gram-Schmidt with the projected vector as float pairs (hi + lo, 48
// bits) on the FP32 pipe.  The stored vectors are exact floats, so every product with one is an
// exact product of floats plus a correction; the sums keep their rounding errors (two-sum), over
// the warp as pairs, over the warps in FP64.  The result is rounded to FP32 as before: its error
// against 64 bits is that rounding either way (8^4, 24 vectors: 2.55e-8, and 7.53e-7 for vectors that
// differ by 1/30, with FP64 arithmetic as with pairs).  Eleven FP32 instructions stand for an
// FP64 one of 1/64 the rate: 16^3 x 32, 24 vectors 11.8 -> 2.2 ms.
DEV void pair_mac(dfloat& a, dfloat w, float q) {   // a += w q
    const float p = __fmul_rn(w.hi, q);
    float e = fmaf(w.hi, q, -p);
    e = fmaf(w.lo, q, e);
    const dfloat t = two_sum(a.hi, p);
    a.hi = t.hi;
    a.lo = __fadd_rn(a.lo, __fadd_rn(t.lo, e));
}
DEV void pair_square(dfloat& a, dfloat w) {   // a += w w
    const float p = __fmul_rn(w.hi, w.hi);
    float e = fmaf(w.hi, w.hi, -p);
    e = fmaf(__fadd_rn(w.hi, w.hi), w.lo, e);
    const dfloat t = two_sum(a.hi, p);
    a.hi = t.hi;
    a.lo = __fadd_rn(a.lo, __fadd_rn(t.lo, e));
}
DEV dfloat shfl_xor_pair(dfloat v, int off) {
    return dfloat(__shfl_xor_sync(0xffffffffu, v.hi, off), __shfl_xor_sync(0xffffffffu, v.lo, off));
}
// sums of four pairs over the warp; lanes 8k .. 8k + 7 get the sum of value transposed_index<4>
DEV dfloat transposed_pair_sum4(dfloat (&v)[4], int lane) {
#pragma unroll
    for (int h = 2, off = 16; h >= 1; h /= 2, off /= 2) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const dfloat keep = up ? v[k + h] : v[k], give = up ? v[k] : v[k + h];
            v[k] = keep + shfl_xor_pair(give, off);
        }
    }
    dfloat r = v[0];
#pragma unroll
    for (int off = 4; off >= 1; off /= 2) r = r + shfl_xor_pair(r, off);
    return r;
}
// |w|^2 of the block (every thread gets it); one pair per warp through red, contains barriers
DEV double pair_norm(const dfloat (&wr)[6], const dfloat (&wi)[6], double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    dfloat n;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        pair_square(n, wr[k]);
        pair_square(n, wi[k]);
    }
    n = quick_two_sum(n.hi, n.lo);
#pragma unroll
    for (int off = 16; off >= 1; off /= 2) n = n + shfl_xor_pair(n, off);
    if (lane == 0) red[warp] = to_double(n);
    __syncthreads();
    double t = 0;
    for (int w = 0; w < nw; ++w) t += red[w];
    __syncthreads();
    return t;
}
__global__ void __launch_bounds__(512) orthonormalise_pairs_kernel(Geom g, Blocking bk, int nvec, void* vecs, int* err) {
    __shared__ double red[32];
    __shared__ float redm[32];
    __shared__ float2 s_inv;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float2* part = reinterpret_cast<float2*>(smem_raw);                    // [nwarps][nvec][re, im] pairs
    float4* coef = reinterpret_cast<float4*>(part + (size_t)nw * nvec * 2);   // [nvec]: re.hi, re.lo, im.hi, im.lo
    const int Xi = blockIdx.x, chi = blockIdx.y;
    const int l = threadIdx.x;
    const bool active = l < bk.Vb;
    const size_t vb = spinor_bytes<P32>(g.V);
    int c[4], s = 0;
    if (active) s = block_site(g, bk, Xi, l, c);
    for (int i = 0; i < nvec; ++i) {
        // w scaled by the power of two that brings its largest component on this domain to [1, 2)
        // (exact, and the result does not depend on it): squares of any FP32 values stay in range
        dfloat wr[6], wi[6];
        cx<float> u0[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) u0[k] = czero<float>();
        if (active) load_chirality<P32>((const char*)vecs + i * vb, g.V, s, chi, u0);
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) m = fmaxf(m, fmaxf(fabsf(u0[k].re), fabsf(u0[k].im)));
#pragma unroll
        for (int off = 16; off >= 1; off /= 2) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        if (lane == 0) redm[warp] = m;
        __syncthreads();
        for (int w = 0; w < nw; ++w) m = fmaxf(m, redm[w]);
        const int e = (int)(__float_as_uint(m) >> 23);   // biased exponent; 0: zero or subnormal
        const float sc = m > 0.f && e < 255 ? __uint_as_float((unsigned)min(253, max(1, 254 - e)) << 23) : 1.f;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            wr[k] = dfloat(sc * u0[k].re);
            wi[k] = dfloat(sc * u0[k].im);
        }
        const double n0 = pair_norm(wr, wi, red);   // its barriers keep redm's readers from the next writers
        double nn = n0;
        for (int pass = 0; pass < 2 && i > 0; ++pass) {
            // a second projection only after a large cancellation
            if (pass == 1 && nn > 0.25 * n0) break;
            for (int j0 = 0; j0 < i; j0 += 2) {
                cx<float> u[2][6];
#pragma unroll
                for (int t = 0; t < 2; ++t)
                    if (active && j0 + t < i) load_chirality<P32>((const char*)vecs + (j0 + t) * vb, g.V, s, chi, u[t]);
                dfloat q[4];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    dfloat re, im;   // <v_j, w>
                    if (active && j0 + t < i) {
#pragma unroll
                        for (int k = 0; k < 6; ++k) {
                            pair_mac(re, wr[k], u[t][k].re);
                            pair_mac(re, wi[k], u[t][k].im);
                            pair_mac(im, wi[k], u[t][k].re);
                            pair_mac(im, wr[k], -u[t][k].im);
                        }
                    }
                    q[2 * t] = quick_two_sum(re.hi, re.lo);
                    q[2 * t + 1] = quick_two_sum(im.hi, im.lo);
                }
                const dfloat tot = transposed_pair_sum4(q, lane);
                const int v = transposed_index<4>(lane);
                if ((lane & 7) == 0 && j0 + (v >> 1) < i)
                    part[((size_t)warp * nvec + j0 + (v >> 1)) * 2 + (v & 1)] = make_float2(tot.hi, tot.lo);
            }
            __syncthreads();
            for (int j = l; j < i; j += blockDim.x) {
                double re = 0, im = 0;
                for (int w = 0; w < nw; ++w) {
                    const float2 a = part[((size_t)w * nvec + j) * 2], b = part[((size_t)w * nvec + j) * 2 + 1];
                    re += (double)a.x + (double)a.y;
                    im += (double)b.x + (double)b.y;
                }
                const dfloat r = split_double(re), m = split_double(im);
                coef[j] = make_float4(r.hi, r.lo, m.hi, m.lo);
            }
            __syncthreads();
            for (int j0 = 0; j0 < i; j0 += 2) {
                cx<float> u[2][6];
#pragma unroll
                for (int t = 0; t < 2; ++t)
                    if (active && j0 + t < i) load_chirality<P32>((const char*)vecs + (j0 + t) * vb, g.V, s, chi, u[t]);
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (!active || j0 + t >= i) break;
                    const float4 cc = coef[j0 + t];   // w -= c v_j
                    const dfloat nr(-cc.x, -cc.y), ni(-cc.z, -cc.w), pi(cc.z, cc.w);
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        pair_mac(wr[k], nr, u[t][k].re);
                        pair_mac(wr[k], pi, u[t][k].im);
                        pair_mac(wi[k], nr, u[t][k].im);
                        pair_mac(wi[k], ni, u[t][k].re);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) {   // the low parts gathered corrections: back to proper pairs
                wr[k] = two_sum(wr[k].hi, wr[k].lo);
                wi[k] = two_sum(wi[k].hi, wi[k].lo);
            }
            nn = pair_norm(wr, wi, red);   // also keeps part / coef readers apart from the next pass
        }
        // rank test: |w| <= 1e-5 |w0| (FP32 storage)
        if (threadIdx.x == 0) {
            double t = nn;
            if (!(t > 1e-10 * n0)) {
                atomicExch(err, 1);
                t = 1.0;
            }
            const dfloat v = split_double(1.0 / sqrt(t));
            s_inv = make_float2(v.hi, v.lo);
        }
        __syncthreads();
        if (active) {
            // the other chirality half belongs to the CTA (Xi, 1 - chi): write ours only
            const dfloat inv(s_inv.x, s_inv.y);
            cx<float> hv[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const dfloat a = inv * wr[k], b = inv * wi[k];
                hv[k] = {a.hi, b.hi};
            }
            SpinorIO<P32>::store_half((char*)vecs + i * vb, g.V, s, chi, hv);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ Galerkin operator
// CTA (block Xi, pair of columns J = (t, j)): for every direction d the fields
// T_d = H_d P_t v_j on the sites of Xi (H_0 = D_SAP on the block, H_{+-mu} =
// the hops of D leaving Xi through its +-mu face) are formed for both columns
// and projected on all basis vectors of Xi: B[Xi][I][d][J] = <Xi, I| T_d>.
// Each test-vector load serves both columns, and the four projections of a
// vector (two columns x two chiralities) are summed over the warp by one
// transposed shuffle reduction.  d = 0 takes one thread per site; a face
// direction has a quarter of the sites (4^4 blocks), so the face's T goes to
// shared memory and the CTA's threads split into groups over the same face
// sites, each group projecting on its share of the test vectors: the vectors
// are read from L2 for 3 blocks' worth of sites per column pair instead of
// 6.5 (every warp has sites of most faces).  The column pairs of a block are
// neighbours in the grid, so that 23 of 24 find its vectors in L2 (blocks first,
// the 302 MB of vectors came from DRAM for every pair, 5.3 TB/s of it).  16^3 x
// 32, 24 vectors: 11.0 -> 3.7 ms; bound by the latency of L2 at 16 warps per SM.
template <class PV, typename TC>
__global__ void __launch_bounds__(PV::id == 0 ? 256 : 512) galerkin_kernel(Geom g, Blocking bk, int nvec, const void* __restrict__ vecs,
                                const void* __restrict__ U, const void* __restrict__ C, typename PV::T kappa,
                                void* B) {
    using T = typename PV::T;
    constexpr int NQ = 8;   // per vector: column a / b x chirality 0 / 1 x (re, im)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nc = 2 * nvec;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T* partf = reinterpret_cast<T*>(smem_raw);   // [nwarps][2 columns][nc] complex
    cx<T>* part = reinterpret_cast<cx<T>*>(smem_raw);
    cx<T>* tsh = part + (size_t)nw * 2 * nc;     // [2 columns][12][face sites, padded]
    // the pairs of one block follow each other: they read the block's vectors from L2
    const int Xi = blockIdx.x / nvec, Ja = 2 * (blockIdx.x % nvec), Jb = Ja + 1;
    const bool hasB = Jb < nc;
    const int ta = Ja / nvec, ja = Ja % nvec, tb = hasB ? Jb / nvec : 0, jb = hasB ? Jb % nvec : 0;
    const size_t vb = spinor_bytes<PV>(g.V);
    const char* va = (const char*)vecs + ja * vb;
    const char* vbp = (const char*)vecs + jb * vb;
    const int qi = transposed_index<NQ>(lane);
    const bool writer = (lane & (32 / NQ - 1)) == 0;
    auto load_proj = [&](const char* v, int t, int site, cx<T> out[12]) {
        SpinorIO<PV>::load(v, g.V, site, out);
#pragma unroll
        for (int k = 0; k < 6; ++k) {   // selects, so that the spinor stays in registers
            if (t != 0) out[k] = czero<T>();
            else out[6 + k] = czero<T>();
        }
    };
    // acc_a += coeff (1 - dir gamma_mu) W P_ta v_ja(n), acc_b likewise (one link load)
    auto hop2 = [&](int n, int linksite, int mu, int dir, T coeff, cx<T> (&acc_a)[12], cx<T> (&acc_b)[12]) {
        cx<T> psi[12], u[3][3];
        GaugeIO<PV>::load(U, g.V, mu, linksite, u);
        load_proj(va, ta, n, psi);
        hop_accum<T>(acc_a, psi, u, mu, dir, coeff);
        if (hasB) {
            load_proj(vbp, tb, n, psi);
            hop_accum<T>(acc_b, psi, u, mu, dir, coeff);
        }
    };
    for (int d = 0; d < 9; ++d) {
        const int mu = d == 0 ? 0 : (d - 1) % 4;
        const int dir = d <= 4 ? +1 : -1;
        // this direction's sites: nf of them, padded to whole warps, and the groups of threads over them
        const int nf = d == 0 ? bk.Vb : bk.Vb / bk.b[mu];
        const int nfp = (nf + 31) / 32 * 32, ngrp = blockDim.x / nfp, nwf = nfp >> 5;
        const int grp = threadIdx.x / nfp, f = threadIdx.x - grp * nfp;
        const bool work = grp < ngrp && f < nf;
        int c[4] = {0, 0, 0, 0}, s = 0;
        cx<T> Ta[12], Tb[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) Ta[k] = Tb[k] = czero<T>();
        if (work) {
            int l = f;
            if (d != 0) {
                int low = 1;
                for (int m = 0; m < mu; ++m) low *= bk.b[m];
                l = f % low + low * ((dir > 0 ? bk.b[mu] - 1 : 0) + bk.b[mu] * (f / low));
            }
            s = block_site(g, bk, Xi, l, c);
        }
        if (work && grp == 0) {
            float ph;
            if (d == 0) {
                cx<T> psi[12];
                load_proj(va, ta, s, psi);
                clover_apply<PV>(C, g.V, s, psi, Ta);
                if (hasB) {
                    load_proj(vbp, tb, s, psi);
                    clover_apply<PV>(C, g.V, s, psi, Tb);
                }
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int lc = c[m] % bk.b[m];
                    if (lc != bk.b[m] - 1) {
                        int n = neighbour(g, s, c, m, +1, ph);
                        hop2(n, s, m, +1, -kappa * T(ph), Ta, Tb);
                    }
                    if (lc != 0) {
                        int n = neighbour(g, s, c, m, -1, ph);
                        hop2(n, n, m, -1, -kappa * T(ph), Ta, Tb);
                    }
                }
            } else {
                // the direction is uniform; unrolled so that the spinors are indexed by constants
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (d == 1 + m) {
                        const int n = neighbour(g, s, c, m, +1, ph);
                        hop2(n, s, m, +1, -kappa * T(ph), Ta, Tb);
                    } else if (d == 5 + m) {
                        const int n = neighbour(g, s, c, m, -1, ph);
                        hop2(n, n, m, -1, -kappa * T(ph), Ta, Tb);
                    }
                }
            }
            if (ngrp > 1) {
#pragma unroll
                for (int k = 0; k < 12; ++k) {
                    tsh[k * nfp + f] = Ta[k];
                    tsh[(12 + k) * nfp + f] = Tb[k];
                }
            }
        }
        if (ngrp > 1) {
            __syncthreads();
            if (work && grp > 0) {
#pragma unroll
                for (int k = 0; k < 12; ++k) {
                    Ta[k] = tsh[k * nfp + f];
                    Tb[k] = tsh[(12 + k) * nfp + f];
                }
            }
        }
        const int wf = warp - grp * nwf;   // warp within its group (groups are whole warps)
        for (int i = grp; i < nvec && grp < ngrp; i += ngrp) {
            cx<T> d0a = czero<T>(), d1a = czero<T>(), d0b = czero<T>(), d1b = czero<T>();
            if (work) {
                cx<T> v[12];
                SpinorIO<PV>::load((const char*)vecs + i * vb, g.V, s, v);
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    cfmac(d0a, v[k], Ta[k]);
                    cfmac(d1a, v[6 + k], Ta[6 + k]);
                    cfmac(d0b, v[k], Tb[k]);
                    cfmac(d1b, v[6 + k], Tb[6 + k]);
                }
            }
            T q[NQ] = {d0a.re, d0a.im, d1a.re, d1a.im, d0b.re, d0b.im, d1b.re, d1b.im};
            const T tot = transposed_warp_sum<NQ>(q, lane);
            if (writer) {
                const int col = qi >> 2, comp = qi & 3;
                const int row = (comp < 2 ? 0 : nvec) + i;
                partf[2 * ((wf * 2 + col) * nc + row) + (comp & 1)] = tot;
            }
        }
        __syncthreads();
        for (int r = threadIdx.x; r < 2 * nc; r += blockDim.x) {
            const int col = r / nc, row = r % nc;
            if (col == 1 && !hasB) continue;
            cx<T> acc = czero<T>();
            for (int w = 0; w < nwf; ++w) acc = acc + part[(w * 2 + col) * nc + row];
            CStore<TC>::st(B, (((size_t)Xi * nc + row) * 9 + d) * nc + (col ? Jb : Ja), ccast<TC>(acc));
        }
        __syncthreads();
    }
}

int threads_for(const Blocking& bk) { return (bk.Vb + 31) / 32 * 32; }

// right-hand sides per CTA: the batch in groups of up to four, as even as they go (FP64 fields
// and blocks of more than 256 sites take one: the registers of four do not fit)
struct RhsSplit {
    int groups, per;
};
RhsSplit split_rhs(int nrhs, int threads, bool many) {
    if (!many || nrhs == 1 || threads > 256) return {nrhs, 1};
    const int groups = (nrhs + 3) / 4;
    return {groups, (nrhs + groups - 1) / groups};
}

template <class PF, class PV, typename TC, class IO = SpinorIO<PF>>
cudaError_t restrict_impl(const GeomH& gh, const BlockH& bh, int nvec, const void* vecs, const void* fine,
                          void* coarse, int nrhs, cudaStream_t st) {
    Geom g = make_geom(gh);
    Blocking bk = make_blocking(gh, bh);
    const int th = threads_for(bk);
    const size_t fstride = spinor_bytes<PF>(g.V);   // canonical and internal FP32 fields have the same size
    const RhsSplit sp = split_rhs(nrhs, th, PF::id != 0 && PV::id != 0);
    const dim3 grid((nrhs + sp.per - 1) / sp.per, std::min(bk.Vc, 65535));
    auto smem = [&](int nb) { return (size_t)(th / 32) * nb * 2 * nvec * sizeof(cx<typename PF::T>); };
    note_launch();
    if constexpr (PF::id != 0 && PV::id != 0) {
        if (sp.per > 2) {
            restrict_batch_kernel<PF, PV, TC, 4, IO><<<grid, th, smem(4), st>>>(g, bk, nvec, vecs, fine, fstride, coarse, nrhs, sp.per);
            return cudaGetLastError();
        }
        if (sp.per == 2) {
            restrict_batch_kernel<PF, PV, TC, 2, IO><<<grid, th, smem(2), st>>>(g, bk, nvec, vecs, fine, fstride, coarse, nrhs, sp.per);
            return cudaGetLastError();
        }
    }
    restrict_kernel<PF, PV, TC, IO><<<grid, th, smem(1), st>>>(g, bk, nvec, vecs, fine, fstride, coarse);
    return cudaGetLastError();
}
template <class PF, class PV, typename TC, class IO = SpinorIO<PF>>
cudaError_t prolong_impl(const GeomH& gh, const BlockH& bh, int nvec, const void* vecs, const void* coarse,
                         void* fine, int nrhs, cudaStream_t st) {
    Geom g = make_geom(gh);
    Blocking bk = make_blocking(gh, bh);
    const int th = threads_for(bk);
    const size_t fstride = spinor_bytes<PF>(g.V);
    const RhsSplit sp = split_rhs(nrhs, th, PF::id != 0 && PV::id != 0);
    const dim3 grid((nrhs + sp.per - 1) / sp.per, std::min(bk.Vc, 65535));
    auto smem = [&](int nb) { return (size_t)nb * 2 * nvec * sizeof(cx<typename PF::T>); };
    note_launch();
    if constexpr (PF::id != 0 && PV::id != 0) {
        if (sp.per > 2) {
            prolong_batch_kernel<PF, PV, TC, 4, IO><<<grid, th, smem(4), st>>>(g, bk, nvec, vecs, coarse, fine, fstride, nrhs, sp.per);
            return cudaGetLastError();
        }
        if (sp.per == 2) {
            prolong_batch_kernel<PF, PV, TC, 2, IO><<<grid, th, smem(2), st>>>(g, bk, nvec, vecs, coarse, fine, fstride, nrhs, sp.per);
            return cudaGetLastError();
        }
    }
    prolong_kernel<PF, PV, TC, IO><<<grid, th, smem(1), st>>>(g, bk, nvec, vecs, coarse, fine, fstride);
    return cudaGetLastError();
}

}  // namespace

#define DISPATCH_F(fprec, ...)                 \
    if (fprec == 0) { using PF = P64; __VA_ARGS__; } \
    else if (fprec == 1) { using PF = P32; __VA_ARGS__; } \
    else { using PF = P16; __VA_ARGS__; }

cudaError_t launch_restrict_fine(int fprec, int vprec, int cprec, const GeomH& g, const BlockH& bk, int nvec,
                                 const void* vecs, const void* fine, void* coarse, int nrhs, cudaStream_t st) {
    if (vprec == 0) {
        if (cprec == 0) { DISPATCH_F(fprec, return restrict_impl<PF, P64, double>(g, bk, nvec, vecs, fine, coarse, nrhs, st)); }
        DISPATCH_F(fprec, return restrict_impl<PF, P64, float>(g, bk, nvec, vecs, fine, coarse, nrhs, st));
    }
    if (vprec == 2) {   // half-precision test vectors with a per-site scale
        if (cprec == 0) { DISPATCH_F(fprec, return restrict_impl<PF, P16, double>(g, bk, nvec, vecs, fine, coarse, nrhs, st)); }
        DISPATCH_F(fprec, return restrict_impl<PF, P16, float>(g, bk, nvec, vecs, fine, coarse, nrhs, st));
    }
    if (cprec == 0) { DISPATCH_F(fprec, return restrict_impl<PF, P32, double>(g, bk, nvec, vecs, fine, coarse, nrhs, st)); }
    DISPATCH_F(fprec, return restrict_impl<PF, P32, float>(g, bk, nvec, vecs, fine, coarse, nrhs, st));
}
cudaError_t launch_prolong_fine(int fprec, int vprec, int cprec, const GeomH& g, const BlockH& bk, int nvec,
                                const void* vecs, const void* coarse, void* fine, int nrhs, cudaStream_t st) {
    if (vprec == 0) {
        if (cprec == 0) { DISPATCH_F(fprec, return prolong_impl<PF, P64, double>(g, bk, nvec, vecs, coarse, fine, nrhs, st)); }
        DISPATCH_F(fprec, return prolong_impl<PF, P64, float>(g, bk, nvec, vecs, coarse, fine, nrhs, st));
    }
    if (vprec == 2) {
        if (cprec == 0) { DISPATCH_F(fprec, return prolong_impl<PF, P16, double>(g, bk, nvec, vecs, coarse, fine, nrhs, st)); }
        DISPATCH_F(fprec, return prolong_impl<PF, P16, float>(g, bk, nvec, vecs, coarse, fine, nrhs, st));
    }
    if (cprec == 0) { DISPATCH_F(fprec, return prolong_impl<PF, P32, double>(g, bk, nvec, vecs, coarse, fine, nrhs, st)); }
    DISPATCH_F(fprec, return prolong_impl<PF, P32, float>(g, bk, nvec, vecs, coarse, fine, nrhs, st));
}
bool transfer_canon_supported(int vprec, int cprec, const void* fine) {
    return vprec != 0 && cprec == 1 && ((uintptr_t)fine & 15) == 0;
}
cudaError_t launch_restrict_canon(int vprec, const GeomH& g, const BlockH& bk, int nvec, const void* vecs,
                                  const void* fine, void* coarse, int nrhs, cudaStream_t st) {
    if (vprec == 2) return restrict_impl<P32, P16, float, CanonF32>(g, bk, nvec, vecs, fine, coarse, nrhs, st);
    return restrict_impl<P32, P32, float, CanonF32>(g, bk, nvec, vecs, fine, coarse, nrhs, st);
}
cudaError_t launch_prolong_canon(int vprec, const GeomH& g, const BlockH& bk, int nvec, const void* vecs,
                                 const void* coarse, void* fine, int nrhs, cudaStream_t st) {
    if (vprec == 2) return prolong_impl<P32, P16, float, CanonF32>(g, bk, nvec, vecs, coarse, fine, nrhs, st);
    return prolong_impl<P32, P32, float, CanonF32>(g, bk, nvec, vecs, coarse, fine, nrhs, st);
}
cudaError_t launch_orthonormalise_fine(int vprec, const GeomH& gh, const BlockH& bh, int nvec, void* vecs,
                                       int* err, cudaStream_t st) {
    Geom g = make_geom(gh);
    Blocking bk = make_blocking(gh, bh);
    dim3 grid(bk.Vc, 2);
    int th = threads_for(bk);
    const size_t smem = ((size_t)(th / 32) + 1) * nvec * sizeof(cx<double>);
    if (vprec == 0) (note_launch(), orthonormalise_kernel<<<grid, th, smem, st>>>(g, bk, nvec, vecs, err));
    else (note_launch(), orthonormalise_pairs_kernel<<<grid, th, smem, st>>>(g, bk, nvec, vecs, err));
    return cudaGetLastError();
}
cudaError_t launch_galerkin_fine(int vprec, int cprec, const GeomH& gh, const BlockH& bh, int nvec, const void* vecs,
                                 const void* U, const void* C, double kappa, void* B, cudaStream_t st) {
    Geom g = make_geom(gh);
    Blocking bk = make_blocking(gh, bh);
    int th = threads_for(bk);
    const unsigned grid = (unsigned)bk.Vc * nvec;   // block, pair of columns (nvec pairs: 2 nvec columns)
    // T of the largest face that leaves room for a second group of threads
    size_t face = 0;
    for (int mu = 0; mu < 4; ++mu) {
        const size_t nfp = (bk.Vb / bk.b[mu] + 31) / 32 * 32;
        if (th >= (int)(2 * nfp) && 24 * nfp > face) face = 24 * nfp;
    }
    // Partial sums and face tile: past the 48 KB that a launch gets unasked for blocks with an extent
    // of two (24 x 256 face sites of FP32 are 48 KB by themselves) and for FP64 blocks of many vectors;
    // 80 KB at 64 vectors on 512 (FP32) or 256 (FP64) threads.  The limit is always set to that bound:
    // a launch from another thread never finds it lowered to a smaller block's need.
    constexpr int kSmemBound = 80 * 1024;
    const size_t smem = ((size_t)(th / 32) * 2 * 2 * nvec + face) * (vprec == 0 ? sizeof(cx<double>) : sizeof(cx<float>));
    auto launch = [&](auto kernel, auto kap) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBound);
        if (e != cudaSuccess) return e;
        (note_launch(), kernel<<<grid, th, smem, st>>>(g, bk, nvec, vecs, U, C, kap, B));
        return cudaGetLastError();
    };
    if (vprec == 0) return cprec == 0 ? launch(galerkin_kernel<P64, double>, kappa) : launch(galerkin_kernel<P64, float>, kappa);
    return cprec == 0 ? launch(galerkin_kernel<P32, double>, (float)kappa)
                      : launch(galerkin_kernel<P32, float>, (float)kappa);
}

// ---------------------------------------------------------------- ragged batches
// blockDim: the largest problem's block, rounded up to whole warps; shared memory for that many warps
cudaError_t launch_restrict_ragged(int vprec, const void* d, const int* off, int np, int ctas, int max_vb, int max_nvec,
                                   cudaStream_t st) {
    const int th = (max_vb + 31) / 32 * 32;
    const size_t smem = (size_t)(th / 32) * 2 * max_nvec * sizeof(cx<float>);
    const RaggedDev* dd = (const RaggedDev*)d;
    if (vprec == 0) (note_launch(), restrict_ragged_kernel<P64><<<ctas, th, smem, st>>>(dd, off, np));
    else if (vprec == 1) (note_launch(), restrict_ragged_kernel<P32><<<ctas, th, smem, st>>>(dd, off, np));
    else (note_launch(), restrict_ragged_kernel<P16><<<ctas, th, smem, st>>>(dd, off, np));
    return cudaGetLastError();
}
cudaError_t launch_prolong_ragged(int vprec, const void* d, const int* off, int np, int ctas, int max_vb, int max_nvec,
                                  cudaStream_t st) {
    const int th = (max_vb + 31) / 32 * 32;
    const size_t smem = (size_t)2 * max_nvec * sizeof(cx<float>);
    const RaggedDev* dd = (const RaggedDev*)d;
    if (vprec == 0) (note_launch(), prolong_ragged_kernel<P64><<<ctas, th, smem, st>>>(dd, off, np));
    else if (vprec == 1) (note_launch(), prolong_ragged_kernel<P32><<<ctas, th, smem, st>>>(dd, off, np));
    else (note_launch(), prolong_ragged_kernel<P16><<<ctas, th, smem, st>>>(dd, off, np));
    return cudaGetLastError();
}

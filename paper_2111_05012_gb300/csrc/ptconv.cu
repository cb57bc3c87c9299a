// Gauge-equivariant parallel-transport convolution layers of the learned
// preconditioner:
//   out^a(x) = sum_b sum_d W_d^{ab} (T_d in^b)(x),
//   T_0 = 1, (T_{+mu} f)(x) = U_mu(x) f(x+mu), (T_{-mu} f)(x) = U_mu(x-mu)^dag f(x-mu)
// (fermion boundary phase on the t wrap), W_d^{ab} a complex 4x4 spin matrix
// stored in bfloat16 and applied with FP32 accumulation.  Fields are FP32
// internal spinors, C channels stored one after another.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int kMaxC = 4;

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
int sms() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

// y = U v (dir > 0) or U^dag v (dir < 0) on the three colours of each spin
DEV void colour_mul(const cx<float> u[3][3], int dir, const cx<float> v[12], cx<float> y[12]) {
    if (dir > 0) {
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                cx<float> t = u[a][0] * v[3 * sp];
                cfma(t, u[a][1], v[3 * sp + 1]);
                cfma(t, u[a][2], v[3 * sp + 2]);
                y[3 * sp + a] = t;
            }
    } else {
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                cx<float> t = cmulc(u[0][a], v[3 * sp]);
                cfmac(t, u[1][a], v[3 * sp + 1]);
                cfmac(t, u[2][a], v[3 * sp + 2]);
                y[3 * sp + a] = t;
            }
    }
}

// What T_d reads at site s, as loaded: the neighbour's spinor, the link (rows 0 and 1) and the
// boundary phase.  Kept raw so that the next direction's loads can be in flight under the
// arithmetic of the current one.
struct HopSite {
    int n, link;   // neighbour, and the site that holds the link
    float ph;
};
DEV HopSite hop_site(const Geom& g, int s, const int c[4], int d) {
    HopSite h = {s, s, 1.f};
    // the direction is the same in every lane; unrolled so that c stays in registers
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        if (d == 1 + mu) h.n = neighbour(g, s, c, mu, 1, h.ph);
        if (d == 5 + mu) h.link = h.n = neighbour(g, s, c, mu, -1, h.ph);
    }
    return h;
}
struct RawSpinor {
    float4 r[6];
    DEV void load(const void* f, int V, int n) {
#pragma unroll
        for (int q = 0; q < 6; ++q) r[q] = __ldg((const float4*)f + (size_t)q * V + n);
    }
    DEV void get(cx<float> v[12]) const {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            v[2 * q] = {r[q].x, r[q].y};
            v[2 * q + 1] = {r[q].z, r[q].w};
        }
    }
};
struct RawLink {
    float4 a, b, c;
    DEV void load(const void* U, int V, int mu, int n) {
        const float4* p = (const float4*)U + (size_t)mu * 3 * V;
        a = __ldg(p + n);
        b = __ldg(p + (size_t)V + n);
        c = __ldg(p + (size_t)2 * V + n);
    }
    DEV void get(float ph, cx<float> u[3][3]) const {
        u[0][0] = {a.x, a.y};
        u[0][1] = {a.z, a.w};
        u[0][2] = {b.x, b.y};
        u[1][0] = {b.z, b.w};
        u[1][1] = {c.x, c.y};
        u[1][2] = {c.z, c.w};
        reconstruct_row2(u);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) u[i][k] = ph * u[i][k];
    }
};
struct RawHop {
    RawSpinor v;
    RawLink l;
    float ph;
    DEV void load(const Geom& g, const void* U, const void* f, int s, const int c[4], int d) {
        const HopSite h = hop_site(g, s, c, d);
        ph = h.ph;
        v.load(f, g.V, h.n);
        if (d > 0) l.load(U, g.V, (d - 1) & 3, h.link);
    }
    // (T_d f)(s), times the power of two sc
    DEV void get(int d, cx<float> out[12], float sc = 1.f) const {
        if (d == 0) {
            v.get(out);
#pragma unroll
            for (int k = 0; k < 12; ++k) out[k] = sc * out[k];
            return;
        }
        cx<float> f[12], u[3][3];
        v.get(f);
        l.get(sc * ph, u);
        colour_mul(u, d <= 4 ? 1 : -1, f, out);
    }
};

// acc += w phi for a complex 4x4 spin matrix w in shared memory (two entries per 16-byte read)
DEV void spin_mac(cx<float> acc[12], const cx<float>* w, const cx<float> phi[12]) {
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int t = 0; t < 4; t += 2) {
            const float4 q = *reinterpret_cast<const float4*>(w + sp * 4 + t);
#pragma unroll
            for (int col = 0; col < 3; ++col) {
                cfma(acc[3 * sp + col], cx<float>{q.x, q.y}, phi[3 * t + col]);
                cfma(acc[3 * sp + col], cx<float>{q.z, q.w}, phi[3 * (t + 1) + col]);
            }
        }
}

// A thread's sum of squares of any FP32 values in FP64: a site's 24 squares on the FP32 pipe, with
// the rounding errors of the products and of the sums kept so that nothing is lost that FP64 would
// hold; the sites in FP64 (FP64 instructions run at 1/64 of the FP32 rate; a site takes six of
// them instead of 48).
// hi and mid start at powers of two c0 and c1 (times 1.5) that no term exceeds, so the three-operation
// quick_two_sum is exact for them: squares are at most c0, the errors of hi and of the products at
// most 2^-19 c0 and all 48 of them together below c1 / 2.  What lo loses is of order 2^-55 c0.
// A site whose largest component lies outside [2^-38, 2^50] is scaled by a power of two first: the
// errors of smaller squares would fall below the FP32 range, larger squares overflow it.
struct SquareSum {
    double d = 0;
    // the 24 components of a site, v(k)
    template <class F> DEV void add(F&& v) {
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 24; ++k) m = fmaxf(m, fabsf(v(k)));
        const float sc = m < 0x1p-38f ? 0x1p80f : m > 0x1p50f ? 0x1p-80f : 1.f;
        const float ms = sc * m;
        const float c0 = __uint_as_float((__float_as_uint(ms * ms) & 0x7f800000u) + 0x00800000u);
        const float c1 = 0x1.8p-12f * c0;
        float hi = c0, mid = c1, lo = 0.f;
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            const float x = sc * v(k), p = __fmul_rn(x, x);
            const dfloat t = quick_two_sum(hi, p), u = quick_two_sum(mid, t.lo);
            const dfloat w = quick_two_sum(u.hi, fmaf(x, x, -p));
            hi = t.hi;
            mid = w.hi;
            lo = __fadd_rn(lo, __fadd_rn(u.lo, w.lo));
        }
        if (!(fabsf(hi) <= 0x1.fffffep127f)) {   // an infinity or a NaN: the error terms would turn both into NaN
            float q = 0.f;
#pragma unroll
            for (int k = 0; k < 24; ++k) q = fmaf(v(k), v(k), q);
            d += q;
            return;
        }
        const double t = ((double)lo + (double)__fsub_rn(mid, c1)) + (double)__fsub_rn(hi, c0);
        d += sc == 1.f ? t : t * (sc > 1.f ? 0x1p-160 : 0x1p160);
    }
    DEV double get() const { return d; }
};

// The last layer of a training pass: y is replaced by y - e for the canonical target e, and
// part[cta] receives the CTA's shares of |y - e|^2 and |e|^2
struct LossArgs {
    const float4* e;   // canonical, 6 float4 per site; null outside training
    double2* part;
};
DEV void loss_site(const LossArgs& l, int s, cx<float> acc[12], SquareSum& d2, SquareSum& e2) {
    float e[24];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const float4 t = __ldg(l.e + (size_t)s * 6 + q);
        acc[2 * q] = acc[2 * q] - cx<float>{t.x, t.y};
        acc[2 * q + 1] = acc[2 * q + 1] - cx<float>{t.z, t.w};
        e[4 * q] = t.x;
        e[4 * q + 1] = t.y;
        e[4 * q + 2] = t.z;
        e[4 * q + 3] = t.w;
    }
    e2.add([&](int k) { return e[k]; });
    d2.add([&](int k) { return k & 1 ? acc[k >> 1].im : acc[k >> 1].re; });
}
DEV void loss_block(const LossArgs& l, const SquareSum& d2, const SquareSum& e2) {
    __shared__ double red[2 * 32];
    double v[2] = {d2.get(), e2.get()};
    block_sum<double, 2>(v, red);
    if (threadIdx.x == 0) l.part[blockIdx.x] = make_double2(v[0], v[1]);
}

// Forward layers.  The colour transport T_d and the spin matrices W_d act on different indices
// and commute, so the layer transports whichever side has fewer channels:
// up (cin <= cout): out^a += W_d^{ab} (T_d in^b), cin transports per direction;
// down (cin > cout): out^a += T_d (sum_b W_d^{ab} in^b), cout transports per direction.
// Bound by the FP32 pipe (16 cin cout 9 complex spin entries x 3 colours per site, the
// transports 8 x 36 complex products per transported channel).  128 threads, so that 160
// registers still leave three CTAs per SM; the loop over the directions stays rolled to keep the
// body in the instruction cache.  24^3 x 48: 1 -> 4 channels 331 -> 258 us, 4 -> 1 501 -> 332 us (loss included).
constexpr int kFT = 128;
DEV void load_weights(cx<float>* w, const __nv_bfloat16* __restrict__ W, int nw) {
    for (int i = threadIdx.x; i < nw; i += blockDim.x)
        w[i] = {__bfloat162float(W[2 * i]), __bfloat162float(W[2 * i + 1])};
    __syncthreads();
}
template <int COUT, bool LOSS>
__global__ void __launch_bounds__(kFT, COUT >= 3 ? 3 : 4) ptconv_up_kernel(Geom g, int cin, const void* __restrict__ U,
                                                            const __nv_bfloat16* __restrict__ W, const void* in,
                                                            void* out, LossArgs loss) {
    __shared__ __align__(16) cx<float> w[COUT * COUT * 9 * 16];   // cin <= COUT
    load_weights(w, W, COUT * cin * 9 * 16);
    const size_t fb = spinor_bytes<P32>(g.V);
    SquareSum d2, e2;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < g.V; s += gridDim.x * blockDim.x) {
        int c[4];
        site_coords(g, s, c);
        cx<float> acc[COUT][12];
#pragma unroll
        for (int a = 0; a < COUT; ++a)
#pragma unroll
            for (int k = 0; k < 12; ++k) acc[a][k] = czero<float>();
        RawHop h;
        h.load(g, U, in, s, c, 0);
#pragma unroll 1
        for (int b = 0, d = 0; b < cin;) {
            cx<float> phi[12];
            h.get(d, phi);
            const cx<float>* wd = w + (b * 9 + d) * 16;
            if (++d == 9) {
                d = 0;
                ++b;
            }
            if (b < cin) h.load(g, U, (const char*)in + b * fb, s, c, d);
#pragma unroll
            for (int a = 0; a < COUT; ++a) spin_mac(acc[a], wd + a * cin * 144, phi);
        }
        if constexpr (LOSS) loss_site(loss, s, acc[0], d2, e2);
#pragma unroll
        for (int a = 0; a < COUT; ++a) SpinorIO<P32>::store((char*)out + a * fb, g.V, s, acc[a]);
    }
    if constexpr (LOSS) loss_block(loss, d2, e2);
}
template <int CIN, bool LOSS>
__global__ void __launch_bounds__(kFT, 3) ptconv_down_kernel(Geom g, int cout, const void* __restrict__ U,
                                                             const __nv_bfloat16* __restrict__ W, const void* in,
                                                             void* out, LossArgs loss) {
    __shared__ __align__(16) cx<float> w[CIN * (CIN > 1 ? CIN - 1 : 1) * 9 * 16];   // cout < CIN
    load_weights(w, W, cout * CIN * 9 * 16);
    const size_t fb = spinor_bytes<P32>(g.V);
    SquareSum d2, e2;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < g.V; s += gridDim.x * blockDim.x) {
        int c[4];
        site_coords(g, s, c);
#pragma unroll 1
        for (int a = 0; a < cout; ++a) {
            cx<float> acc[12];
#pragma unroll
            for (int k = 0; k < 12; ++k) acc[k] = czero<float>();
            RawSpinor r;
            r.load(in, g.V, s);
#pragma unroll 1
            for (int d = 0; d < 9; ++d) {
                const HopSite h = hop_site(g, s, c, d);
                RawLink l;
                if (d > 0) l.load(U, g.V, (d - 1) & 3, h.link);
                cx<float> v[12];
#pragma unroll
                for (int k = 0; k < 12; ++k) v[k] = czero<float>();
#pragma unroll
                for (int b = 0; b < CIN; ++b) {
                    cx<float> f[12];
                    r.get(f);
                    // the next channel, or the next direction's first
                    if (b + 1 < CIN) r.load((const char*)in + (b + 1) * fb, g.V, h.n);
                    else if (d < 8) r.load(in, g.V, hop_site(g, s, c, d + 1).n);
                    spin_mac(v, w + ((a * CIN + b) * 9 + d) * 16, f);
                }
                if (d > 0) {
                    cx<float> u[3][3], y[12];
                    l.get(h.ph, u);
                    colour_mul(u, d <= 4 ? 1 : -1, v, y);
#pragma unroll
                    for (int k = 0; k < 12; ++k) acc[k] = acc[k] + y[k];
                } else {
#pragma unroll
                    for (int k = 0; k < 12; ++k) acc[k] = v[k];
                }
            }
            if constexpr (LOSS) loss_site(loss, s, acc, d2, e2);
            SpinorIO<P32>::store((char*)out + a * fb, g.V, s, acc);
        }
    }
    if constexpr (LOSS) loss_block(loss, d2, e2);
}

// Weight gradient G[a][b][d][s][t] = sum_{x,c} gout^a(x)[s,c] conj((T_d in^b)(x)[t,c]); since
// T_d^dag = T_rev(d), it is also sum (T_rev(d) gout^a)[s,c] conj(in^b[t,c]) (ADJ), and the side
// with fewer channels is the one transported.  A warp has all NS x 16 sums of one direction in
// registers, its lanes over the sites; the eight warps of a CTA take the eight hops of the same
// sites, so the NS static fields come from L1 for seven of them (with one CTA per direction they
// were re-read nine times from L2 or DRAM).  The first n0 CTAs take d = 0, their warps different
// sites.  Eight warps, not nine: with nine one SM quarter holds three and the registers per
// thread fall from 255 to 168, which spills the sums.  The next sites' loads are in flight under
// the products.  blockIdx.y: the transported channel.
// Every kFlush sites per lane the sums move on, over the warp, into float pairs (48 bits), so
// the plain FP32 accumulation is no longer than a few sites.  24^3 x 48, four static channels:
// 1 -> 4 layer 757 -> 479 us, 4 -> 1 layer 1140 -> 459 us; bound by the FP32 pipe and by latency
// at eight warps per SM.
// part[(blockIdx.y * 9 + d) * max(gridDim.x - n0, n0) + cta][NS * 16]
constexpr int kWT = 256, kFlush = 8;
// Power of two on the transported side of a training pair of very small or large targets: in and
// y - e scale alike, and their FP32 products would leave the range long before the fields do
DEV float grad_scale(const double2* __restrict__ norm) {
    if (!norm || !(norm->y > 0) || (norm->y >= 0x1p-60 && norm->y <= 0x1p80)) return 1.f;
    return (float)exp2((double)max(-120, min(120, -ilogb(norm->y) / 2)));
}
template <int NS, bool ADJ>
__global__ void __launch_bounds__(kWT, 1) ptconv_wgrad_kernel(Geom g, const void* __restrict__ U, const void* moved,
                                                              const void* fixed, int n0, double2* part,
                                                              const double2* __restrict__ norm) {
    const float psc = grad_scale(norm);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool self = (int)blockIdx.x < n0;
    const int d = self ? 0 : warp + 1;
    const int td = !ADJ || d == 0 ? d : (d <= 4 ? d + 4 : d - 4);
    // this warp's stretches of 32 sites: first + k * step
    const int cta = self ? blockIdx.x : blockIdx.x - n0, ncta = self ? n0 : gridDim.x - n0;
    const int first = self ? (cta * 8 + warp) * 32 : cta * 32, step = self ? ncta * 256 : ncta * 32;
    const size_t fb = spinor_bytes<P32>(g.V);
    const char* mv = (const char*)moved + blockIdx.y * fb;
    float acc[NS][32];
    dfloat tot[NS];
#pragma unroll
    for (int a = 0; a < NS; ++a)
#pragma unroll
        for (int k = 0; k < 32; ++k) acc[a][k] = 0.f;
    auto flush = [&]() {
#pragma unroll
        for (int a = 0; a < NS; ++a) {
            const float t = transposed_warp_sum<32>(acc[a], lane);
            const dfloat q = two_sum(tot[a].hi, t);
            tot[a].hi = q.hi;
            tot[a].lo = __fadd_rn(tot[a].lo, q.lo);
#pragma unroll
            for (int k = 0; k < 32; ++k) acc[a][k] = 0.f;
        }
    };
    RawHop h;
    auto fetch = [&](int s) {
        if (s < g.V) {
            int c[4];
            site_coords(g, s, c);
            h.load(g, U, mv, s, c, td);
        }
    };
    fetch(first + lane);
    int it = 0;
    // s0 is uniform over the warp: lanes past the last site take part in the sums with zeros
    for (int s0 = first; s0 < g.V; s0 += step) {
        const int s = s0 + lane;
        if (s < g.V) {
            RawSpinor r;
            r.load(fixed, g.V, s);
            cx<float> phi[12];
            h.get(td, phi, psc);
            fetch(s + step);
#pragma unroll
            for (int a = 0; a < NS; ++a) {
                cx<float> f[12];
                r.get(f);
                if (a + 1 < NS) r.load((const char*)fixed + (a + 1) * fb, g.V, s);
#pragma unroll
                for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        cx<float> q = {acc[a][2 * (4 * sp + t)], acc[a][2 * (4 * sp + t) + 1]};
#pragma unroll
                        for (int col = 0; col < 3; ++col) {
                            if constexpr (ADJ) cfmac(q, f[3 * t + col], phi[3 * sp + col]);
                            else cfmac(q, phi[3 * t + col], f[3 * sp + col]);
                        }
                        acc[a][2 * (4 * sp + t)] = q.re;
                        acc[a][2 * (4 * sp + t) + 1] = q.im;
                    }
            }
        }
        if (++it == kFlush) {
            flush();
            it = 0;
        }
    }
    flush();
    const int qi = transposed_index<32>(lane);
    const int per = max((int)gridDim.x - n0, n0);
    double* const pd = reinterpret_cast<double*>(part);
    if (!self) {
        double* o = pd + ((size_t)(blockIdx.y * 9 + d) * per + cta) * (NS * 32);
#pragma unroll
        for (int a = 0; a < NS; ++a) o[a * 32 + qi] = to_double(tot[a]);
        return;
    }
    // d = 0: the eight warps' sums of the CTA, in order
    __shared__ double red[NS * 32][9];
#pragma unroll
    for (int a = 0; a < NS; ++a) red[a * 32 + qi][warp] = to_double(tot[a]);
    __syncthreads();
    for (int q = threadIdx.x; q < NS * 32; q += kWT) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += red[q][w];
        pd[((size_t)(blockIdx.y * 9) * per + cta) * (NS * 32) + q] = t;
    }
}

// the CTAs' partial sums in a fixed order, one warp per complex entry:
// G[a][b][d][k] (+)= sum / |e|^2 (norm: the pair (|y - e|^2, |e|^2) of the training pair, or null)
__global__ void __launch_bounds__(256) ptconv_wsum_kernel(int cin, int ns, int nmoved, int adj, int n0,
                                                          int n8, const double2* __restrict__ part,
                                                          const double2* __restrict__ norm, int add, double2* G) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);   // (moved channel, d, fixed channel, k)
    if (i >= nmoved * 9 * ns * 16) return;
    const int q = i % (ns * 16), md = i / (ns * 16), d = md % 9, m = md / 9;
    double re = 0, im = 0;
    const int ncta = d == 0 ? n0 : n8, per = max(n0, n8);
    for (int k = lane; k < ncta; k += 32) {
        const double2 v = part[((size_t)md * per + k) * (ns * 16) + q];
        re += v.x;
        im += v.y;
    }
    re = warp_sum(re);
    im = warp_sum(im);
    if (lane == 0) {
        const int a = adj ? m : q / 16, b = adj ? q / 16 : m;
        double2& o = G[(((size_t)a * cin + b) * 9 + d) * 16 + q % 16];
        const double sc = (norm ? 1.0 / norm->y : 1.0) / grad_scale(norm);
        o = make_double2((add ? o.x : 0.0) + sc * re, (add ? o.y : 0.0) + sc * im);
    }
}
// norms[pair] = sum of the CTAs' shares of (|y - e|^2, |e|^2)
__global__ void __launch_bounds__(32) loss_sum_kernel(const double2* __restrict__ part, int ncta, double2* out) {
    double a = 0, b = 0;
    for (int k = threadIdx.x; k < ncta; k += 32) {
        a += part[k].x;
        b += part[k].y;
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if (threadIdx.x == 0) *out = make_double2(a, b);
}

}  // namespace

size_t ptconv_partials(int cin, int cout) {
    // weight-gradient partials of a layer, or the loss shares of its CTAs
    const size_t w = (size_t)cin * cout * 9 * 16 * sms();
    const size_t l = (size_t)sms() * 16;
    return w > l ? w : l;
}

cudaError_t launch_ptconv_forward(const GeomH& gh, int cin, int cout, const void* U32, const void* Wbf16,
                                  const void* in, void* out, cudaStream_t st, const float* target, double2* part,
                                  double2* norms) {
    if (cin < 1 || cin > kMaxC || cout < 1 || cout > kMaxC || (target && cout != 1)) return cudaErrorInvalidValue;
    Geom g = make_geom(gh);
    int grid = (g.V + kFT - 1) / kFT;
    if (grid > sms() * 16) grid = sms() * 16;
    const __nv_bfloat16* W = (const __nv_bfloat16*)Wbf16;
    const LossArgs l = {(const float4*)target, part};
#define UP(C, L) (note_launch(), ptconv_up_kernel<C, L><<<grid, kFT, 0, st>>>(g, cin, U32, W, in, out, l))
#define DOWN(C, L) (note_launch(), ptconv_down_kernel<C, L><<<grid, kFT, 0, st>>>(g, cout, U32, W, in, out, l))
    if (cin <= cout) {
        switch (cout) {
            case 1: if (target) UP(1, true); else UP(1, false); break;
            case 2: UP(2, false); break;
            case 3: UP(3, false); break;
            default: UP(4, false); break;
        }
    } else {
        switch (cin) {
            case 2: if (target) DOWN(2, true); else DOWN(2, false); break;
            case 3: if (target) DOWN(3, true); else DOWN(3, false); break;
            default: if (target) DOWN(4, true); else DOWN(4, false); break;
        }
    }
#undef UP
#undef DOWN
    if (target) (note_launch(), loss_sum_kernel<<<1, 32, 0, st>>>(part, grid, norms));
    return cudaGetLastError();
}

cudaError_t launch_ptconv_wgrad(const GeomH& gh, int cin, int cout, const void* U32, const void* in,
                                const void* gout, double2* part, const double2* norm, bool add, double2* G,
                                cudaStream_t st) {
    if (cin < 1 || cin > kMaxC || cout < 1 || cout > kMaxC) return cudaErrorInvalidValue;
    Geom g = make_geom(gh);
    const bool adj = cin > cout;   // transport gout instead of in
    const int nm = adj ? cout : cin, ns = adj ? cin : cout;
    // eight hops on one set of CTAs, d = 0 (a tenth of the work: no transport, one direction) on
    // another; together one CTA per SM
    const int need = (g.V + 31) / 32, n8 = std::min(need, std::max(1, sms() - sms() / 10));
    const int n0 = std::min((need + 7) / 8, std::max(1, sms() / 10));
    const dim3 grid(n0 + n8, nm);
#define WG(N, A) (note_launch(), ptconv_wgrad_kernel<N, A><<<grid, kWT, 0, st>>>(g, U32, A ? gout : in, A ? in : gout, n0, part, norm))
    switch (ns) {
        case 1: WG(1, false); break;
        case 2: if (adj) WG(2, true); else WG(2, false); break;
        case 3: if (adj) WG(3, true); else WG(3, false); break;
        default: if (adj) WG(4, true); else WG(4, false); break;
    }
#undef WG
    const int n = nm * 9 * ns * 16;
    (note_launch(), ptconv_wsum_kernel<<<(n + 7) / 8, 256, 0, st>>>(cin, ns, nm, adj, n0, n8, part, norm, add, G));
    return cudaGetLastError();
}

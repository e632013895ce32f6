// Learned right preconditioner M: a linear, gauge-equivariant parallel-transport
// convolution network with channels 1 -> 12 -> 1, no activation (so M is linear).
//
//   layer: out[c](x) = sum_{k=0..8} sum_{c'} W[k, c, c'] (T_k in[c'])(x)
//   T_0 = 1, T_{1+d} with d = 2 mu: U_mu(x) f(x+mu); d = 2 mu + 1: U_mu(x-mu)^+ f(x-mu)
//
// The transport of site x in direction d uses exactly the gathered link d of
// the hop kernels (hop_impl.cuh) and the same boundary phases. W[k, c, c'] is
// a complex 4x4 matrix on spin. M maps an even-site vector to an even-site
// vector: layer 1 fans the single input channel out to 12 hidden channels on
// all sites, layer 2 folds them back onto the even sites.
//
// Weights (flat float layout shared with the C ABI): W1[k][c][s][t][re,im]
// then W2[k][c][s][t][re,im], 9 * 12 * 16 complex each. The kernels read them
// as given (the library stores BF16-rounded values for the solver).
//
// Training: for L = sum |M v - y|^2/|y|^2 + mu |A M v - v|^2/|v|^2 the weight
// gradients dL/dRe W + i dL/dIm W follow from the 8 x 8 (+ 1) correlations of
// the transported loss gradient with the transported input (below).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "blas_impl.cuh"
#include "chunk.h"
#include "handle.h"

namespace wd {

constexpr int PTC_C = 12;                 // hidden channels
constexpr int PTC_LAYER = 9 * PTC_C * 16; // complex weights per layer
constexpr int PTC_FLOATS = 2 * PTC_LAYER * 2;

// Link d of site h (gathered layout, R reals of LT) as 18 floats (row 2 rebuilt for R = 12).
template <typename LT, int R>
__device__ __forceinline__ void load_link(const uint4* __restrict__ links, int Vh, int h, int d, float (&m)[18]) {
    constexpr int N = Unit<LT>::N;
#pragma unroll
    for (int e = 0; e < R; ++e) {
        const int el = d * R + e;
        const uint4 w = __ldg(links + (size_t)(el / N) * Vh + h);
        m[e] = (float)Unit<LT>::get(w, el % N);
    }
    if (R == 12) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int b1 = (b + 1) % 3, b2 = (b + 2) % 3;
            const float ar = m[2 * b1], ai = m[2 * b1 + 1], br = m[6 + 2 * b2], bi = m[6 + 2 * b2 + 1];
            const float cr = m[2 * b2], ci = m[2 * b2 + 1], dr = m[6 + 2 * b1], di = m[6 + 2 * b1 + 1];
            m[12 + 2 * b] = ar * br - ai * bi - cr * dr + ci * di;
            m[12 + 2 * b + 1] = -(ar * bi + ai * br - cr * di - ci * dr);
        }
    }
}

// phi = m f on colour for each of the 4 spins (f, phi: [spin][colour][re,im]);
// each output is one multiply and a chain of fused multiply-adds.
__device__ __forceinline__ void colour_mul(const float (&m)[18], const float (&f)[24], float (&phi)[24]) {
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float* mr = &m[6 * a];
            const float* fs = &f[6 * s];
            float re = mr[0] * fs[0];
            re = __fmaf_rn(-mr[1], fs[1], re);
            re = __fmaf_rn(mr[2], fs[2], re);
            re = __fmaf_rn(-mr[3], fs[3], re);
            re = __fmaf_rn(mr[4], fs[4], re);
            re = __fmaf_rn(-mr[5], fs[5], re);
            float im = mr[0] * fs[1];
            im = __fmaf_rn(mr[1], fs[0], im);
            im = __fmaf_rn(mr[2], fs[3], im);
            im = __fmaf_rn(mr[3], fs[2], im);
            im = __fmaf_rn(mr[4], fs[5], im);
            im = __fmaf_rn(mr[5], fs[4], im);
            phi[2 * (3 * s + a)] = re;
            phi[2 * (3 * s + a) + 1] = im;
        }
}

// acc += w phi on spin (w: 16 complex [s][t] as float2 in shared memory).
__device__ __forceinline__ void spin_mul_add_p(const float2* w, const float* phi, float (&acc)[24]) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float fr = phi[2 * (3 * t + a)], fi = phi[2 * (3 * t + a) + 1];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const float2 c = w[4 * s + t];
                acc[2 * (3 * s + a)] = __fmaf_rn(-c.y, fi, __fmaf_rn(c.x, fr, acc[2 * (3 * s + a)]));
                acc[2 * (3 * s + a) + 1] = __fmaf_rn(c.y, fr, __fmaf_rn(c.x, fi, acc[2 * (3 * s + a) + 1]));
            }
        }
}
// The same on FP32x2 pairs (re, im), term for term: w holds (c.x, c.x, -c.y, c.y), phi and acc complex numbers.
__device__ __forceinline__ void spin_mul_add_x2(const float4* w, const float2* phi, float2 (&acc)[12]) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        float2 f[3], g[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f[a] = phi[3 * t + a];
            g[a] = make_float2(f[a].y, f[a].x);
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const float4 c = w[4 * s + t];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                acc[3 * s + a] = __ffma2_rn(make_float2(c.z, c.w), g[a],
                                            __ffma2_rn(make_float2(c.x, c.y), f[a], acc[3 * s + a]));
        }
    }
}
__device__ __forceinline__ void spin_mul_add(const float2* w, const float (&phi)[24], float (&acc)[24]) {
    spin_mul_add_p(w, phi, acc);
}

// ---------------------------------------------------------- collapsed M ---
//
// The network has no nonlinearity and its spin weights commute with the
// colour transports, so its two layers collapse exactly:
//   M psi = sum_{k2} T_{k2} phi_{k2},  phi_{k2} = sum_{k1} V[k2][k1] T_{k1} psi,
//   V[k2][k1] = sum_c W2[k2][c] W1[k1][c]   (4x4 spin matrix products).
// For an even-site input (odd sites zero) only phi_0 = V[0][0] psi on the
// even sites and phi_{1+d} (d = 0..7) on the odd sites are nonzero, so M is
// two stencil passes with eight odd-site intermediate fields instead of the
// twelve hidden channels on both parities.

// V[k2][k1][s][t] from the BF16-rounded weights (double accumulation).
__global__ void k_ptc_collapse(const float* w, float2* V) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 81 * 16; i += gridDim.x * blockDim.x) {
        const int k2 = i / 144, k1 = (i / 16) % 9, s = (i / 4) % 4, t = i % 4;
        double re = 0.0, im = 0.0;
        for (int c = 0; c < PTC_C; ++c)
            for (int u = 0; u < 4; ++u) {
                const float* a = w + 2 * PTC_LAYER + 2 * ((k2 * PTC_C + c) * 16 + 4 * s + u);
                const float* b = w + 2 * ((k1 * PTC_C + c) * 16 + 4 * u + t);
                re += (double)a[0] * b[0] - (double)a[1] * b[1];
                im += (double)a[0] * b[1] + (double)a[1] * b[0];
            }
        V[i] = make_float2((float)re, (float)im);
    }
}

constexpr int S1_SITES = 32;                // sites per block of the first pass
constexpr int S1_STRIDE = 8 * 24 + 2;       // floats per site of its transport tile (padded, pairs aligned)

// First pass on the odd sites y: the eight transports T_{1+d} psi(y) (warp mu
// computes directions 2 mu and 2 mu + 1 for the block's 32 sites) go to shared
// memory; then warp mu forms phi_{1+d}(y) = sum_{k1} V[1+d][k1] T_{k1} psi(y)
// for its two directions and stores them.
template <typename TIN, typename TPHI, typename LT, int R>
__global__ void __launch_bounds__(128) k_ptc_s1(Geom g, const uint4* in_e, uint4* phi, long long pvs,
                                                const uint4* links_o, const float2* V, const SolverState* guard) {
    if (guarded(guard, GUARD_INNER)) return;
    in_e += blockIdx.y * (long long)Spinor<TIN>::UNITS * g.Vh;      // sample blockIdx.y, vectors back to back
    phi += blockIdx.y * 8 * pvs;
    __shared__ __align__(16) float ts[S1_SITES * S1_STRIDE];
    __shared__ float4 vs[64 * 16];   // V[1 + a][1 + b] at 16 (8 a + b), as spin_mul_add_x2 takes it
    for (int i = threadIdx.x; i < 64 * 16; i += blockDim.x) {
        const float2 c = V[((1 + i / 128) * 9 + 1 + (i / 16) % 8) * 16 + i % 16];
        vs[i] = make_float4(c.x, c.x, -c.y, c.y);
    }
    __syncthreads();
    const int mu = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* mine = ts + lane * S1_STRIDE;
    for (int base = blockIdx.x * S1_SITES; base < g.Vh; base += gridDim.x * S1_SITES) {
        const int h = base + lane;
        const bool ok = h < g.Vh;
        if (ok) {
            const Coord co = coord_of(g, 1, h);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int d = 2 * mu + j;
                bool wrap;
                const int hn = neighbour(g, h, co, d, &wrap);
                float f[24], m[18], t[24];
                load_spinor<TIN>(in_e, g.Vh, hn, f);
                if (wrap && g.bc[mu] < 0) {
#pragma unroll
                    for (int i = 0; i < 24; ++i) f[i] = -f[i];
                }
                load_link<LT, R>(links_o, g.Vh, h, d, m);
                colour_mul(m, f, t);
#pragma unroll
                for (int i = 0; i < 24; ++i) mine[d * 24 + i] = t[i];
            }
        }
        __syncthreads();
        if (ok) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int d2 = 2 * mu + j;
                float2 sum[12];
#pragma unroll
                for (int i = 0; i < 12; ++i) sum[i] = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int k1 = 0; k1 < 8; ++k1)
                    spin_mul_add_x2(&vs[16 * (8 * d2 + k1)], reinterpret_cast<const float2*>(mine + 24 * k1), sum);
                float acc[24];
#pragma unroll
                for (int i = 0; i < 12; ++i) {
                    acc[2 * i] = sum[i].x;
                    acc[2 * i + 1] = sum[i].y;
                }
                store_spinor<TPHI>(phi + (size_t)d2 * pvs, g.Vh, h, acc);
            }
        }
        __syncthreads();
    }
}

// The 2 units of gathered-link storage that hold link d of a site (12 halves
// of an FP16 12-real link start at element 12 d), and the link rebuilt from them.
template <typename LT> __device__ __forceinline__ void load_link_units(const uint4* __restrict__ links, int Vh, int h,
                                                                       int d, uint4 (&u)[2]) {
    const int base = (12 * d) / Unit<LT>::N;
    u[0] = __ldg(links + (size_t)base * Vh + h);
    u[1] = __ldg(links + (size_t)(base + 1) * Vh + h);
}
template <typename LT> __device__ __forceinline__ void link_from_units(const uint4 (&u)[2], int d, float (&m)[18]) {
    constexpr int N = Unit<LT>::N;
    const int base = (12 * d) / N;
#pragma unroll
    for (int e = 0; e < 12; ++e) {
        const int el = 12 * d + e;
        m[e] = (float)Unit<LT>::get(u[el / N - base], el % N);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {   // row 2 = conj(row 0 x row 1)
        const int b1 = (b + 1) % 3, b2 = (b + 2) % 3;
        float re = m[2 * b2 + 1] * m[6 + 2 * b1 + 1];
        re = __fmaf_rn(-m[2 * b2], m[6 + 2 * b1], re);
        re = __fmaf_rn(-m[2 * b1 + 1], m[6 + 2 * b2 + 1], re);
        re = __fmaf_rn(m[2 * b1], m[6 + 2 * b2], re);
        float nim = m[2 * b2] * m[6 + 2 * b1 + 1];
        nim = __fmaf_rn(m[2 * b2 + 1], m[6 + 2 * b1], nim);
        nim = __fmaf_rn(-m[2 * b1], m[6 + 2 * b2 + 1], nim);
        nim = __fmaf_rn(-m[2 * b1 + 1], m[6 + 2 * b2], nim);
        m[12 + 2 * b] = re;
        m[12 + 2 * b + 1] = nim;
    }
}

// Second pass of the FP16 path with colour-major phi (as the tensor-core first
// pass writes it): every direction's phi units and link units are loaded one
// direction ahead of the arithmetic that uses them.
template <typename TIN, typename TPHI, typename TOUT, typename LT>
__global__ void __launch_bounds__(128, 5) k_ptc_s2_pf(Geom g, const uint4* in_e, const uint4* phi, long long pvs,
                                                      uint4* out_e, const uint4* links_e, const float2* V,
                                                      const SolverState* guard) {
    if (guarded(guard, GUARD_INNER)) return;
    __shared__ float2 v00[16];
    if (threadIdx.x < 16) v00[threadIdx.x] = V[threadIdx.x];
    __syncthreads();
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < g.Vh; h += gridDim.x * blockDim.x) {
        int nbr[8];
        const unsigned wm = site_neighbours(g, 0, h, nbr);
        uint4 fu[2][3], lu[2][2];
#pragma unroll
        for (int a = 0; a < 3; ++a) fu[0][a] = __ldg(phi + (size_t)a * g.Vh + nbr[0]);
        load_link_units<LT>(links_e, g.Vh, h, 0, lu[0]);
        float acc[24], f[24];
#pragma unroll
        for (int i = 0; i < 24; ++i) acc[i] = 0.f;
        load_spinor<TIN>(in_e, g.Vh, h, f);
        spin_mul_add(v00, f, acc);
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            if (d + 1 < 8) {
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    fu[(d + 1) & 1][a] = __ldg(phi + (size_t)(d + 1) * pvs + (size_t)a * g.Vh + nbr[d + 1]);
                load_link_units<LT>(links_e, g.Vh, h, d + 1, lu[(d + 1) & 1]);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int e = 0; e < 8; ++e) f[2 * (3 * (e >> 1) + a) + (e & 1)] = Unit<TPHI>::get(fu[d & 1][a], e);
            float m[18], t[24];
            link_from_units<LT>(lu[d & 1], d, m);
            colour_mul(m, f, t);
            const float ph = (((wm >> d) & 1u) && g.bc[d >> 1] < 0) ? -1.f : 1.f;
#pragma unroll
            for (int i = 0; i < 24; ++i) acc[i] = __fmaf_rn(ph, t[i], acc[i]);
        }
        store_spinor<TOUT>(out_e, g.Vh, h, acc);
    }
}

// Second pass on the even sites x: M psi(x) = V[0][0] psi(x) + sum_d T_{1+d} phi_{1+d}(x).
template <typename TIN, typename TPHI, typename TOUT, typename LT, int R>
__global__ void __launch_bounds__(128) k_ptc_s2(Geom g, const uint4* in_e, const uint4* phi, long long pvs,
                                                uint4* out_e, const uint4* links_e, const float2* V,
                                                const SolverState* guard) {
    if (guarded(guard, GUARD_INNER)) return;
    in_e += blockIdx.y * (long long)Spinor<TIN>::UNITS * g.Vh;      // sample blockIdx.y, as in k_ptc_s1
    phi += blockIdx.y * 8 * pvs;
    out_e += blockIdx.y * (long long)Spinor<TOUT>::UNITS * g.Vh;
    __shared__ float2 v00[16];
    if (threadIdx.x < 16) v00[threadIdx.x] = V[threadIdx.x];
    __syncthreads();
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < g.Vh; h += gridDim.x * blockDim.x) {
        const Coord co = coord_of(g, 0, h);
        float acc[24], f[24];
#pragma unroll
        for (int i = 0; i < 24; ++i) acc[i] = 0.f;
        load_spinor<TIN>(in_e, g.Vh, h, f);
        spin_mul_add(v00, f, acc);
#pragma unroll 1
        for (int d = 0; d < 8; ++d) {
            bool wrap;
            const int hn = neighbour(g, h, co, d, &wrap);
            float m[18], t[24];
            load_spinor<TPHI>(phi + (size_t)d * pvs, g.Vh, hn, f);
            load_link<LT, R>(links_e, g.Vh, h, d, m);
            colour_mul(m, f, t);
            const float ph = (wrap && g.bc[d >> 1] < 0) ? -1.f : 1.f;
#pragma unroll
            for (int i = 0; i < 24; ++i) acc[i] = __fmaf_rn(ph, t[i], acc[i]);
        }
        store_spinor<TOUT>(out_e, g.Vh, h, acc);
    }
}

}  // namespace wd

#include "ptc_tc.cuh"

namespace wd {

// --------------------------------------------------------------- training ---
//
// With g = 2 dL/dconj(M v) on the even sites, the gradients of both layers are
// small products of the weights with one set of 4 x 4 spin matrices,
//   C[k][k'] = sum over sites and colours of (T_kbar g) (x) conj(T_k' v),  kbar the opposite hop of k,
//   dW2[k][c] = sum_k' C[k][k'] W1[k'][c]^+,   dW1[k'][c] = sum_k W2[k][c]^+ C[k][k'],
// because the hidden channels are H_c = sum_k' W1[k'][c] T_k' v and a transport
// moves from one side of the colour contraction to the other as its adjoint.
// The transports of v and g live on the odd sites (k, k' = 1..8), k = k' = 0 on
// the even ones; all other C vanish. So no hidden channel is formed: M v comes
// from the collapsed network and C is one contraction over 3 V/2 (site, colour)
// rows with 32 x 32 complex results.

constexpr int CORR_SITES = 32;                       // odd sites per tile
constexpr int CORR_ROW = 34;                         // complex numbers per tile row (32, padded: conflict-free writes)
constexpr int CORR_SMEM = 2 * 3 * CORR_SITES * CORR_ROW * (int)sizeof(float2);
constexpr int CORR_FLOATS = 2 * 32 * 32;             // C[1 + d][1 + d'][s][t] as rows (d, s), columns (d', t)

// C over the odd sites of nb samples, each block's sum to its own slot of
// `part`. Per tile of 32 sites warp mu computes directions 2 mu and 2 mu + 1 of
// both fields (the link and the neighbour index once for both) into shared
// memory as rows (site, colour) x 32 complex; then 64 threads per half of the
// rows hold 4 x 4 complex results each in registers. Bound by the FP32 pipe:
// 14.6k multiply-adds per site and sample.
__global__ void __launch_bounds__(128, 4) k_ptc_corr(Geom g, int nb, const uint4* v, const uint4* gr, long long vs,
                                                     const uint4* links_o, float* part) {
    extern __shared__ __align__(16) unsigned char corr_smem[];
    float2* A = reinterpret_cast<float2*>(corr_smem);               // T_kbar g: column 4 d + s
    float2* B = A + 3 * CORR_SITES * CORR_ROW;                      // T_k' v: column 4 d' + t
    const int tid = threadIdx.x, mu = tid >> 5, lane = tid & 31;
    const int half = tid >> 6, r = (tid & 63) >> 3, c = tid & 7;
    float re[4][4], im[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) re[i][j] = im[i][j] = 0.f;
    const int tiles = (g.Vh + CORR_SITES - 1) / CORR_SITES;
    for (int t = blockIdx.x; t < nb * tiles; t += gridDim.x) {
        const int sample = t / tiles, h = (t - sample * tiles) * CORR_SITES + lane;
        const uint4 *vi = v + sample * vs, *gi = gr + sample * vs;
        const bool ok = h < g.Vh;
        const Coord co = ok ? coord_of(g, 1, h) : Coord{};
#pragma unroll 1
        for (int j = 0; j < 2; ++j) {
            const int d = 2 * mu + j;
            float fv[24], fg[24];
            if (ok) {
                bool wrap;
                const int hn = neighbour(g, h, co, d, &wrap);
                float f[24], m[18];
                load_link<float, 18>(links_o, g.Vh, h, d, m);
                if (wrap && g.bc[mu] < 0) {
#pragma unroll
                    for (int i = 0; i < 18; ++i) m[i] = -m[i];
                }
                load_spinor<float>(vi, g.Vh, hn, f);
                colour_mul(m, f, fv);
                load_spinor<float>(gi, g.Vh, hn, f);
                colour_mul(m, f, fg);
            } else {
#pragma unroll
                for (int i = 0; i < 24; ++i) fv[i] = fg[i] = 0.f;
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                float4* pb = reinterpret_cast<float4*>(B + (3 * lane + a) * CORR_ROW + 4 * d);
                float4* pa = reinterpret_cast<float4*>(A + (3 * lane + a) * CORR_ROW + 4 * (d ^ 1));
#pragma unroll
                for (int s = 0; s < 4; s += 2) {
                    const int e = 2 * (3 * s + a), e2 = e + 6;
                    pb[s / 2] = make_float4(fv[e], fv[e + 1], fv[e2], fv[e2 + 1]);
                    pa[s / 2] = make_float4(fg[e], fg[e + 1], fg[e2], fg[e2 + 1]);
                }
            }
        }
        __syncthreads();
        const float4* pa = reinterpret_cast<const float4*>(A + half * 48 * CORR_ROW + 4 * r);
        const float4* pb = reinterpret_cast<const float4*>(B + half * 48 * CORR_ROW + 4 * c);
#pragma unroll 2
        for (int k = 0; k < 48; ++k, pa += CORR_ROW / 2, pb += CORR_ROW / 2) {
            const float4 a0 = pa[0], a1 = pa[1], b0 = pb[0], b1 = pb[1];
            const float ar[4] = {a0.x, a0.z, a1.x, a1.z}, ai[4] = {a0.y, a0.w, a1.y, a1.w};
            const float br[4] = {b0.x, b0.z, b1.x, b1.z}, bi[4] = {b0.y, b0.w, b1.y, b1.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {   // a conj(b)
                    re[i][j] = __fmaf_rn(ai[i], bi[j], __fmaf_rn(ar[i], br[j], re[i][j]));
                    im[i][j] = __fmaf_rn(-ar[i], bi[j], __fmaf_rn(ai[i], br[j], im[i][j]));
                }
        }
        __syncthreads();
    }
    float4* sum = reinterpret_cast<float4*>(corr_smem) + 8 * (tid & 63);   // the second half's share
    if (half == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            sum[2 * i] = make_float4(re[i][0], im[i][0], re[i][1], im[i][1]);
            sum[2 * i + 1] = make_float4(re[i][2], im[i][2], re[i][3], im[i][3]);
        }
    }
    __syncthreads();
    if (half == 0) {
        float4* out = reinterpret_cast<float4*>(part + (size_t)blockIdx.x * CORR_FLOATS);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 w = sum[2 * i + q];
                out[(4 * r + i) * 16 + 2 * c + q] =
                    make_float4(re[i][2 * q] + w.x, im[i][2 * q] + w.y, re[i][2 * q + 1] + w.z, im[i][2 * q + 1] + w.w);
            }
    }
}

// sum[i] (+)= sum over blocks of part[block][i] for `n` floats a block, in a fixed order, as FP32 pairs.
__global__ void __launch_bounds__(256) k_ptc_corr_sum(int blocks, int n, const float* part, int add, float* sum) {
    __shared__ float2 sh[8][32];
    const int i = blockIdx.x * 32 + (threadIdx.x & 31), q = threadIdx.x >> 5;
    F2 t = {0.f, 0.f};
#pragma unroll 16
    for (int b = q; b < blocks; b += 8) t = f2_add(t, F2{part[(size_t)b * n + i], 0.f});
    sh[q][threadIdx.x & 31] = make_float2(t.hi, t.lo);
    __syncthreads();
    if (q == 0) {
        if (add) t = f2_add(t, F2{sum[i], 0.f});
        for (int w = 1; w < 8; ++w) t = f2_add(t, F2{sh[w][threadIdx.x].x, sh[w][threadIdx.x].y});
        sum[i] = t.hi;
    }
}

// Gradients of both layers from C (rows (d, s), columns (d', t)) and C[0][0] (4 x 4): one complex element a thread.
__global__ void k_ptc_wgrad(const float2* C, const float2* C00, const float2* w, float2* grad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * PTC_LAYER) return;
    const int layer = i / PTC_LAYER, e = i % PTC_LAYER;
    const int k = e / (PTC_C * 16), c = (e / 16) % PTC_C, s = (e / 4) % 4, t = e % 4;
    const float2* w1 = w + c * 16;                   // W1[k'][c] at + k' PTC_C 16
    const float2* w2 = w + PTC_LAYER + c * 16;
    float re = 0.f, im = 0.f;
    const int n = k == 0 ? 1 : 8;
    for (int q = 0; q < n; ++q) {
        const int kq = k == 0 ? 0 : 1 + q;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float2 a, b;                             // += a conj(b)
            if (layer == 1) {                        // dW2[k][s][t] = sum C[k][k'][s][u] conj(W1[k'][t][u])
                a = k == 0 ? C00[4 * s + u] : C[(4 * (k - 1) + s) * 32 + 4 * q + u];
                b = w1[kq * PTC_C * 16 + 4 * t + u];
            } else {                                 // dW1[k'][s][t] = sum conj(W2[k][u][s]) C[k][k'][u][t]
                a = k == 0 ? C00[4 * u + t] : C[(4 * q + u) * 32 + 4 * (k - 1) + t];
                b = w2[kq * PTC_C * 16 + 4 * u + s];
            }
            re = __fmaf_rn(a.x, b.x, __fmaf_rn(a.y, b.y, re));
            im = __fmaf_rn(a.y, b.x, __fmaf_rn(-a.x, b.y, im));
        }
    }
    grad[i] = make_float2(re, im);
}

// x^2 added to the FP32 pair s: the square's rounding error is kept.
__device__ __forceinline__ void add_square(F2& s, float x) {
    const float p = __fmul_rn(x, x);
    s = f2_add(s, F2{p, __fmaf_rn(x, x, -p)});
}
// Whether the squares of q, their rounding errors and their sum over any lattice stay in FP32's range.
__device__ __forceinline__ bool ordinary(float x) {
    const float a = fabsf(x);
    return (a >= 0x1p-50f && a <= 0x1p50f) || x == 0.f;
}
__device__ __forceinline__ bool ordinary(const float4& q) {
    return ordinary(q.x) && ordinary(q.y) && ordinary(q.z) && ordinary(q.w);
}

// For sample blockIdx.y: t = gamma5 e2 with e2 = a - v (a = A m), and this
// block's share of |v|^2, |y|^2, |m - y|^2, |e2|^2 (FP32 pairs, about 48 bits; in FP64 the values outside the
// range of FP32 squares).
__global__ void __launch_bounds__(256) k_ptc_resid(int Vh, long long vs, const float4* v, const float4* y,
                                                   const float4* m, const float4* a, float4* t, double* part) {
    const long long o = blockIdx.y * vs;
    F2 s[4] = {};
    double far[4] = {0.0, 0.0, 0.0, 0.0};
    bool any = false;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < vs; i += (long long)gridDim.x * blockDim.x) {
        const float4 vv = v[o + i], yv = y[o + i], mv = m[o + i], av = a[o + i];
        const float4 e1 = make_float4(mv.x - yv.x, mv.y - yv.y, mv.z - yv.z, mv.w - yv.w);
        const float4 e2 = make_float4(av.x - vv.x, av.y - vv.y, av.z - vv.z, av.w - vv.w);
        // (g5 f)_s = -f_{s xor 2}: spins 0, 1 are units 0..2 of a site, spins 2, 3 units 3..5
        t[o + (i < vs / 2 ? i + vs / 2 : i - vs / 2)] = make_float4(-e2.x, -e2.y, -e2.z, -e2.w);
        const float4 q[4] = {vv, yv, e1, e2};
        if (ordinary(vv) && ordinary(yv) && ordinary(e1) && ordinary(e2)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                add_square(s[k], q[k].x);
                add_square(s[k], q[k].y);
                add_square(s[k], q[k].z);
                add_square(s[k], q[k].w);
            }
        } else {
            any = true;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                far[k] = fma((double)q[k].x, (double)q[k].x, far[k]);
                far[k] = fma((double)q[k].y, (double)q[k].y, far[k]);
                far[k] = fma((double)q[k].z, (double)q[k].z, far[k]);
                far[k] = fma((double)q[k].w, (double)q[k].w, far[k]);
            }
        }
    }
    block_sum<4>(s);
    if (__syncthreads_or(any)) block_sum<4>(far);
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k)
            part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + k] = ((double)s[k].hi + (double)s[k].lo) + far[k];
}

// dots[sample][4] = the sums of k_ptc_resid over its nb blocks, in a fixed order (one warp per sample).
__global__ void k_ptc_dots(int nb, const double* part, double* dots) {
    const double* p = part + (size_t)blockIdx.x * nb * 4;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nb; b += 32)
        for (int k = 0; k < 4; ++k) s[k] += p[4 * b + k];
    block_sum<4>(s);
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) dots[4 * blockIdx.x + k] = s[k];
}

// g = 2 (m - y) / |y|^2 + 2 mu gamma5 b / |v|^2 (b = A gamma5 e2) for sample blockIdx.y, and this block's share of
// C[0][0] = sum g (x) conj(v) over the even sites, 32 floats per block.
__global__ void __launch_bounds__(128) k_ptc_lossgrad(int Vh, long long vs, const uint4* v, const uint4* y,
                                                      const uint4* m, const uint4* b, const double* dots, double mu,
                                                      uint4* gr, float* part) {
    const long long o = blockIdx.y * vs;
    const float cy = (float)(2.0 / dots[4 * blockIdx.y + 1]), cv = (float)(2.0 * mu / dots[4 * blockIdx.y]);
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < Vh; h += gridDim.x * blockDim.x) {
        float f[24], e[24], gv[24];
        load_spinor<float>(m + o, Vh, h, e);
        load_spinor<float>(y + o, Vh, h, f);
#pragma unroll
        for (int i = 0; i < 24; ++i) gv[i] = cy * (e[i] - f[i]);
        load_spinor<float>(b + o, Vh, h, f);
#pragma unroll
        for (int i = 0; i < 24; ++i) gv[i] = __fmaf_rn(-cv, f[(i + 12) % 24], gv[i]);
        store_spinor<float>(gr + o, Vh, h, gv);
        load_spinor<float>(v + o, Vh, h, f);
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
                for (int a = 0; a < 3; ++a) {   // g_{s,a} conj(v_{t,a})
                    const float xr = gv[2 * (3 * s + a)], xi = gv[2 * (3 * s + a) + 1];
                    const float yr = f[2 * (3 * t + a)], yi = f[2 * (3 * t + a) + 1];
                    acc[2 * (4 * s + t)] = __fmaf_rn(xi, yi, __fmaf_rn(xr, yr, acc[2 * (4 * s + t)]));
                    acc[2 * (4 * s + t) + 1] = __fmaf_rn(-xr, yi, __fmaf_rn(xi, yr, acc[2 * (4 * s + t) + 1]));
                }
    }
    __shared__ float sh[32][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        float x = acc[i];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
        if (lane == 0) sh[i][warp] = x;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        float x = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) x += sh[threadIdx.x][w];
        part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 32 + threadIdx.x] = x;
    }
}

// Adam on the master weights, then the BF16-rounded copy used by the kernels.
__global__ void k_adam(int n, float* w, const float* g, float* m, float* v, float lr, float b1, float b2, float eps,
                       float c1, float c2, float* weff) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        m[i] = b1 * m[i] + (1.f - b1) * gi;
        v[i] = b2 * v[i] + (1.f - b2) * gi * gi;
        w[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
        weff[i] = __bfloat162float(__float2bfloat16_rn(w[i]));
    }
}

__global__ void k_round_bf16(int n, const float* w, float* weff) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        weff[i] = __bfloat162float(__float2bfloat16_rn(w[i]));
}

// ------------------------------------------------------------------- host ---

static int grid_for(int n, int block) {
    int g = (n + block - 1) / block;
    const int cap = num_sms() * 8;
    return g < 1 ? 1 : (g > cap ? cap : g);
}

struct PtcBufs {
    float *w, *weff, *m, *v, *grad;
    float2* V;      // collapsed spin weights V[k2][k1][s][t] of weff
};

static int ptc_bufs(wd_handle* h, PtcBufs* b) {
    const size_t nb = sizeof(float) * PTC_FLOATS;
    b->w = (float*)workspace(h, "ptc.w", nb);
    b->weff = (float*)workspace(h, "ptc.weff", nb);
    b->m = (float*)workspace(h, "ptc.m", nb);
    b->v = (float*)workspace(h, "ptc.v", nb);
    b->grad = (float*)workspace(h, "ptc.grad", nb);
    b->V = (float2*)workspace(h, "ptc.V", sizeof(float2) * 81 * 16);
    if (!b->w || !b->weff || !b->m || !b->v || !b->grad || !b->V)
        return fail(h, WD_ERR_CUDA, "out of device memory");
    return WD_OK;
}

// Whether the first pass of the FP16 path of M mixes channels on the tensor
// cores (environment WD_PTC_TC=0 selects the FP32-core kernel).
static bool ptc_tensor_cores() {
    static int v = -1;
    if (v < 0) {
        const char* e = std::getenv("WD_PTC_TC");
        v = (e && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Intermediate fields phi_{1+d} of the collapsed M: 8 odd-site vectors in the
// storage type of `prec` (FP32 for WD_FP32, BF16 otherwise).
static uint4* ptc_phi(wd_handle* h, int prec) {
    return prec == WD_FP32 ? (uint4*)workspace(h, "ptc.phi32", vec_bytes(h, WD_FP32) * 8)
                           : (uint4*)workspace(h, "ptc.phi16", vec_bytes(h, WD_BF16) * 8);
}


// M on n FP32 vectors back to back (PHI: 8 vectors each).
static cudaError_t ptc_apply_f32(wd_handle* h, int n, const uint4* in_e, uint4* out_e, uint4* PHI, const float2* V,
                                 const uint4* le, const uint4* lo, cudaStream_t s,
                                 const SolverState* guard = nullptr) {
    const Geom& g = h->g;
    const long long groups = ((long long)g.Vh + S1_SITES - 1) / S1_SITES, cap = (long long)num_sms() * 6;
    const long long pvs = (long long)spinor_units(WD_FP32) * g.Vh;
    k_ptc_s1<float, float, float, 18><<<dim3((int)std::min(groups, cap), n), 128, 0, s>>>(g, in_e, PHI, pvs, lo, V,
                                                                                          guard);
    k_ptc_s2<float, float, float, float, 18><<<dim3(grid_for(g.Vh, 128), n), 128, 0, s>>>(
        g, in_e, PHI, pvs, out_e, le, V, guard);
    return cudaGetLastError();
}

cudaError_t ptc_apply_m(wd_handle* h, int prec, const uint4* in_e, uint4* out_e, uint4* PHI, const float2* V,
                        const uint4* le, const uint4* lo, cudaStream_t s, const SolverState* guard, int* err) {
    const Geom& g = h->g;
    long long groups = ((long long)g.Vh + S1_SITES - 1) / S1_SITES;
    const long long cap = (long long)num_sms() * 6;
    const int g1 = (int)(groups < cap ? groups : cap);
    const int g2 = grid_for(g.Vh, 128);
    if (prec == WD_FP32) {
        return ptc_apply_f32(h, 1, in_e, out_e, PHI, V, le, lo, s, guard);
    } else if (ptc_tensor_cores()) {
        const long long pvs = (long long)spinor_units(WD_BF16) * g.Vh;
        static bool attr = false;
        if (!attr) {
            cudaError_t e = cudaFuncSetAttribute(k_ptc_s1_tc<__half, __half, 12>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM_BYTES);
            if (e != cudaSuccess) return e;
            attr = true;
        }
        const long long tiles = ((long long)g.Vh + tc::TILE_M - 1) / tc::TILE_M;
        const long long tcap = (long long)num_sms() * 3;
        const int gt = (int)(tiles < tcap ? tiles : tcap);
        k_ptc_s1_tc<__half, __half, 12><<<gt, 128, tc::SMEM_BYTES, s>>>(g, in_e, PHI, pvs, lo, V, guard, err,
                                                                         h->wait_rounds);
        k_ptc_s2_pf<__half, __nv_bfloat16, __half, __half><<<g2, 128, 0, s>>>(g, in_e, PHI, pvs, out_e, le, V, guard);
    } else {
        const long long pvs = (long long)spinor_units(WD_BF16) * g.Vh;
        k_ptc_s1<__half, __nv_bfloat16, __half, 12><<<g1, 128, 0, s>>>(g, in_e, PHI, pvs, lo, V, guard);
        k_ptc_s2<__half, __nv_bfloat16, __half, __half, 12><<<g2, 128, 0, s>>>(g, in_e, PHI, pvs, out_e, le, V,
                                                                                        guard);
    }
    return cudaGetLastError();
}

// FP32 even-odd operator A (or A^+ = g5 A g5) on FP32 18-real links, n vectors back to back.
static cudaError_t apply_A_f32(wd_handle* h, int n, const uint4* in, uint4* out, uint4* tmp, const uint4* le,
                               const uint4* lo, cudaStream_t s) {
    HopParams P{};
    P.g = h->g;
    P.nrhs = n;
    P.vs = (long long)spinor_units(WD_FP32) * h->g.Vh;
    P.parity = 1;
    P.links = lo;
    P.in = in;
    P.out = tmp;
    P.a = 1.0;
    cudaError_t e = Ops<float>::hop(18, EPI_H, RED_NONE, P, s);
    if (e != cudaSuccess) return e;
    P.parity = 0;
    P.links = le;
    P.in = tmp;
    P.out = out;
    P.y = in;
    P.a = -h->kappa * h->kappa;
    P.b = 1.0;
    return Ops<float>::hop(18, EPI_Y, RED_NONE, P, s);
}

// Bytes of workspace of a chunk of samples (13 vectors each); a larger batch goes through chunk by chunk. The samples
// of a chunk are gridDim.y of its launches, at most 65535.
constexpr size_t PTC_CHUNK_BYTES = (size_t)2 << 30;
constexpr size_t PTC_CHUNK_SAMPLES = 65535;

int ptc_grad(wd_handle* h, int n, const float* v, const float* y, double mu, double* loss, cudaStream_t s) {
    PtcBufs B;
    int rc = ptc_bufs(h, &B);
    if (rc != WD_OK) return rc;
    const uint4 *le, *lo;
    if ((rc = ensure_links(h, WD_FP32, 18, &le, &lo)) != WD_OK) return rc;
    const Geom& g = h->g;
    const size_t vb = vec_bytes(h, WD_FP32);
    const long long vs = (long long)spinor_units(WD_FP32) * g.Vh;   // 16-byte units of a vector
    const int want = (int)std::max<size_t>(1, std::min<size_t>({(size_t)n, PTC_CHUNK_BYTES / (13 * vb), PTC_CHUNK_SAMPLES}));
    const int rb = (int)std::max<long long>(1, std::min<long long>((vs + 255) / 256, 128));      // blocks per sample
    uint4 *m, *am, *t1, *t2, *gv, *phi;
    double *dots, *dpart;
    float *cpart, *c0part, *C;
    int gb = 0, cb = 0;
    const int chunk = largest_chunk(
        want,
        [&](int c) {
            m = (uint4*)workspace(h, "ptc.vm", vb * c);
            am = (uint4*)workspace(h, "ptc.vam", vb * c);
            t1 = (uint4*)workspace(h, "ptc.vt1", vb * c);
            t2 = (uint4*)workspace(h, "ptc.vt2", vb * c);
            gv = (uint4*)workspace(h, "ptc.vg", vb * c);
            phi = (uint4*)workspace(h, "ptc.phi32", vb * 8 * c);
            gb = std::max(1, std::min((g.Vh + 127) / 128, std::max(1, 4 * num_sms() / c)));
            cb = (int)std::min<long long>((long long)c * ((g.Vh + CORR_SITES - 1) / CORR_SITES), 4 * num_sms());
            dots = (double*)workspace(h, "ptc.dots", sizeof(double) * 4 * (size_t)n);
            dpart = (double*)workspace(h, "ptc.dpart", sizeof(double) * 4 * (size_t)rb * c);
            cpart = (float*)workspace(h, "ptc.cpart", sizeof(float) * (size_t)CORR_FLOATS * cb);
            c0part = (float*)workspace(h, "ptc.c0part", sizeof(float) * 32 * (size_t)gb * c);
            C = (float*)workspace(h, "ptc.C", sizeof(float) * (CORR_FLOATS + 32));
            return m && am && t1 && t2 && gv && phi && dots && dpart && cpart && c0part && C;
        },
        [&]() {
            for (const char* name : {"ptc.vm", "ptc.vam", "ptc.vt1", "ptc.vt2", "ptc.vg", "ptc.phi32"}) drop_workspace(h, name);
            cudaGetLastError();   // the failed allocation's
        });
    if (chunk == 0) return fail(h, WD_ERR_CUDA, "out of device memory");
    static bool attr = false;
    if (!attr) {
        WD_CUDA(h, cudaFuncSetAttribute(k_ptc_corr, cudaFuncAttributeMaxDynamicSharedMemorySize, CORR_SMEM));
        attr = true;
    }
    for (int i0 = 0; i0 < n; i0 += chunk) {
        const int nb = std::min(chunk, n - i0);
        const uint4* vi = reinterpret_cast<const uint4*>(v) + i0 * vs;
        const uint4* yi = reinterpret_cast<const uint4*>(y) + i0 * vs;
        // m = M v ; e2 = A m - v ; b = A gamma5 e2 ; g = 2 (m - y) / |y|^2 + 2 mu gamma5 b / |v|^2
        WD_CUDA(h, ptc_apply_f32(h, nb, vi, m, phi, B.V, le, lo, s));
        WD_CUDA(h, apply_A_f32(h, nb, m, am, t1, le, lo, s));
        k_ptc_resid<<<dim3(rb, nb), 256, 0, s>>>(g.Vh, vs, (const float4*)vi, (const float4*)yi, (const float4*)m,
                                                 (const float4*)am, (float4*)t2, dpart);
        k_ptc_dots<<<nb, 32, 0, s>>>(rb, dpart, dots + 4 * i0);
        WD_CUDA(h, apply_A_f32(h, nb, t2, am, t1, le, lo, s));
        k_ptc_lossgrad<<<dim3(gb, nb), 128, 0, s>>>(g.Vh, vs, vi, yi, m, am, dots + 4 * i0, mu, gv, c0part);
        k_ptc_corr_sum<<<1, 256, 0, s>>>(gb * nb, 32, c0part, i0 > 0, C + CORR_FLOATS);
        const int blocks = (int)std::min<long long>((long long)nb * ((g.Vh + CORR_SITES - 1) / CORR_SITES), cb);
        k_ptc_corr<<<blocks, 128, CORR_SMEM, s>>>(g, nb, vi, gv, vs, lo, cpart);
        k_ptc_corr_sum<<<CORR_FLOATS / 32, 256, 0, s>>>(blocks, CORR_FLOATS, cpart, i0 > 0, C);
        WD_CUDA(h, cudaGetLastError());
    }
    k_ptc_wgrad<<<(2 * PTC_LAYER + 127) / 128, 128, 0, s>>>((const float2*)C, (const float2*)(C + CORR_FLOATS),
                                                            (const float2*)B.weff, (float2*)B.grad);
    WD_CUDA(h, cudaGetLastError());
    std::vector<double> hd(4 * (size_t)n);
    WD_CUDA(h, cudaMemcpyAsync(hd.data(), dots, sizeof(double) * hd.size(), cudaMemcpyDeviceToHost, s));
    WD_CUDA(h, cudaStreamSynchronize(s));
    double L = 0.0;
    for (int i = 0; i < n; ++i) L += hd[4 * i + 2] / hd[4 * i + 1] + mu * hd[4 * i + 3] / hd[4 * i];
    if (loss) *loss = L;
    return WD_OK;
}

}  // namespace wd

using namespace wd;

extern "C" int wd_precond_set(wd_handle* h, const float* w, int where) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (!w || (where != WD_HOST && where != WD_DEVICE)) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_set: bad argument");
    PtcBufs B;
    int rc = ptc_bufs(h, &B);
    if (rc != WD_OK) return rc;
    const size_t nb = sizeof(float) * PTC_FLOATS;
    WD_CUDA(h, cudaMemcpy(B.w, w, nb, where == WD_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice));
    WD_CUDA(h, cudaMemset(B.m, 0, nb));
    WD_CUDA(h, cudaMemset(B.v, 0, nb));
    k_round_bf16<<<(PTC_FLOATS + 255) / 256, 256>>>(PTC_FLOATS, B.w, B.weff);
    k_ptc_collapse<<<6, 256>>>(B.weff, B.V);
    WD_CUDA(h, cudaGetLastError());
    WD_CUDA(h, cudaDeviceSynchronize());
    h->have_precond = true;
    h->adam_t = 0;
    return WD_OK;
}

extern "C" int wd_precond_get(wd_handle* h, float* w, int where) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (!w || (where != WD_HOST && where != WD_DEVICE)) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_get: bad argument");
    if (!h->have_precond) return fail(h, WD_ERR_INVALID_ARG, "no preconditioner weights loaded");
    PtcBufs B;
    int rc = ptc_bufs(h, &B);
    if (rc != WD_OK) return rc;
    WD_CUDA(h, cudaMemcpy(w, B.w, sizeof(float) * PTC_FLOATS,
                          where == WD_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice));
    return WD_OK;
}

extern "C" int wd_precond_apply(wd_handle* h, int prec, const void* in, void* out, void* stream) {
    if (!h) return WD_ERR_INVALID_ARG;
    if ((prec != WD_FP32 && prec != WD_FP16) || !in || !out || in == out)
        return fail(h, WD_ERR_INVALID_ARG, "wd_precond_apply: bad argument");
    if (h->g.part) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_apply: a split lattice (wd_dd_set_partition) has only the wd_dd_* operators");
    if (!h->have_precond) return fail(h, WD_ERR_INVALID_ARG, "no preconditioner weights loaded");
    PtcBufs B;
    int rc = ptc_bufs(h, &B);
    if (rc != WD_OK) return rc;
    const uint4 *le, *lo;
    if ((rc = ensure_links(h, prec, prec == WD_FP32 ? 18 : 12, &le, &lo)) != WD_OK) return rc;
    uint4* PHI = ptc_phi(h, prec);
    int* err = lower_err(h);
    if (!PHI || !err) return fail(h, WD_ERR_CUDA, "out of device memory");
    cudaStream_t s = (cudaStream_t)stream;
    WD_CUDA(h, ptc_apply_m(h, prec, (const uint4*)in, (uint4*)out, PHI, B.V, le, lo, s, nullptr, err));
    WD_CUDA(h, cudaStreamSynchronize(s));
    if (*(volatile int*)h->herr) return fail(h, WD_ERR_TIMEOUT, "wd_precond_apply: a bounded tensor-core wait gave up");
    return WD_OK;
}

extern "C" int wd_precond_grad(wd_handle* h, int n, const float* v, const float* y, double mu, float* grad,
                               double* loss, void* stream) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (n < 1 || !v || !y || !(mu >= 0)) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_grad: bad argument");
    if (h->g.part) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_grad: a split lattice (wd_dd_set_partition) has only the wd_dd_* operators");
    if (!h->have_precond) return fail(h, WD_ERR_INVALID_ARG, "no preconditioner weights loaded");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = ptc_grad(h, n, v, y, mu, loss, s);
    if (rc != WD_OK) return rc;
    if (grad) {
        PtcBufs B;
        if ((rc = ptc_bufs(h, &B)) != WD_OK) return rc;
        WD_CUDA(h, cudaMemcpyAsync(grad, B.grad, sizeof(float) * PTC_FLOATS, cudaMemcpyDeviceToDevice, s));
        WD_CUDA(h, cudaStreamSynchronize(s));
    }
    return WD_OK;
}

extern "C" int wd_precond_train_step(wd_handle* h, int n, const float* v, const float* y, double mu, double lr,
                                     double* loss, void* stream) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (n < 1 || !v || !y || !(mu >= 0) || !(lr > 0)) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_train_step: bad argument");
    if (h->g.part) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_train_step: a split lattice (wd_dd_set_partition) has only the wd_dd_* operators");
    if (!h->have_precond) return fail(h, WD_ERR_INVALID_ARG, "no preconditioner weights loaded");
    cudaStream_t s = (cudaStream_t)stream;
    int rc = ptc_grad(h, n, v, y, mu, loss, s);
    if (rc != WD_OK) return rc;
    PtcBufs B;
    if ((rc = ptc_bufs(h, &B)) != WD_OK) return rc;
    h->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)h->adam_t), c2 = 1.f - std::pow(b2, (float)h->adam_t);
    k_adam<<<(PTC_FLOATS + 255) / 256, 256, 0, s>>>(PTC_FLOATS, B.w, B.grad, B.m, B.v, (float)lr, b1, b2, 1e-8f, c1,
                                                   c2, B.weff);
    k_ptc_collapse<<<6, 256, 0, s>>>(B.weff, B.V);
    WD_CUDA(h, cudaGetLastError());
    WD_CUDA(h, cudaStreamSynchronize(s));
    return WD_OK;
}

// The same weights given as BF16 values in host memory: each widened exactly to FP32 (the BF16 bits are the
// high half of the FP32 word) and loaded as the FP32 masters.
extern "C" int wd_precond_load(wd_handle* h, const void* weights_bf16, size_t n) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (!weights_bf16 || n != (size_t)PTC_FLOATS)
        return fail(h, WD_ERR_INVALID_ARG, "wd_precond_load: n must be WD_PRECOND_FLOATS");
    const unsigned short* b = static_cast<const unsigned short*>(weights_bf16);
    std::vector<float> w(PTC_FLOATS);
    for (size_t i = 0; i < n; ++i) {
        const unsigned u = (unsigned)b[i] << 16;
        std::memcpy(&w[i], &u, sizeof u);
    }
    return wd_precond_set(h, w.data(), WD_HOST);
}

// `steps` Adam steps on the same samples; *loss receives the loss before the last step.
extern "C" int wd_precond_train(wd_handle* h, int steps, int n, const float* v, const float* y, double mu, double lr,
                                double* loss, void* stream) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (steps < 1) return fail(h, WD_ERR_INVALID_ARG, "wd_precond_train: steps must be at least 1");
    double l = 0.0;
    for (int i = 0; i < steps; ++i) {
        const int rc = wd_precond_train_step(h, n, v, y, mu, lr, &l, stream);
        if (rc != WD_OK) return rc;
    }
    if (loss) *loss = l;
    return WD_OK;
}

namespace wd {
// Collapsed spin weights of the loaded network (device), or null when none are loaded.
const float2* ptc_collapsed(wd_handle* h) {
    if (!h->have_precond) return nullptr;
    PtcBufs B;
    if (ptc_bufs(h, &B) != WD_OK) return nullptr;
    return B.V;
}

// Intermediate fields of the collapsed M for the FP16 solve path.
uint4* ptc_phi16(wd_handle* h) { return ptc_phi(h, WD_FP16); }
}  // namespace wd

// Clover (Sheikholeslami-Wohlert) blocks of the Wilson-clover matrix
// D_sw = C - kappa H, the diagonal blocks D_ee = C_ee, D_oo = C_oo of Eqs. 4-5:
//   C(x) = 1 - c_sw kappa sum_{mu<nu} sigma_mu_nu (x) Fh_mu_nu(x),
//   sigma_mu_nu = (i/2) [gamma_mu, gamma_nu],
//   Fh_mu_nu = traceless part of (Q_mu_nu - Q_mu_nu^+) / (8 i),
// Q_mu_nu(x) the four plaquettes of the mu-nu plane with a corner at x, each
// traversed mu-then-nu. Built once per gauge field; C - 1 and C^-1 are stored
// in FP64 in the chiral packing (two Hermitian 6 x 6 blocks, 80 reals per site;
// see mat_mul_chiral), other precisions are made from it on first use. C - 1
// rather than C, since the packing forms the elements that connect opposite
// chiralities as differences of the two blocks' elements: with the 1 in them
// they would be held to the rounding of 1.
//
// In the chiral combinations the spin matrices are Pauli matrices:
// sigma_ij = -eps_ijk sigma_k and sigma_k4 = -(off-diagonal) sigma_k, so block
// c (sg = -1, +1) is
//   S = 1/2 + T,   T = (c_sw kappa / 2) sum_k sigma_k (x) G_k,   G = (F_12 + sg F_03, -F_02 + sg F_13, F_01 + sg F_23)
// (directions 0..3 = x, y, z, t), the packing of
// C - 1 is T and that of C^-1 is S^-1 / 4.
#include <algorithm>
#include <cmath>
#include <string>
#include <type_traits>

#include "fixed64.cuh"
#include "handle.h"
#include "herm6.cuh"

namespace wd {

namespace {

template <typename R> struct Vec3 {
    R v[6];   // three complex numbers
};

// The links of a site as matrices of the products below. FIXED: the gathered
// FP64 links as fixed-point digits (SU(3) links), vectors 64-bit integers in
// units of 2^-59 (fixed64.cuh; the products' magnitudes stay at or below 2);
// otherwise the FP64 links in the host layout and FP64 arithmetic.
struct Field {
    const double* U;
    const uint4* l[2];
    long long V;
    int Vh;
};
struct Site {
    int lex, p;   // lexicographic index and parity
};

template <bool FIXED> struct Links;

template <> struct Links<true> {
    typedef long long R;
    static __device__ __forceinline__ const uint4* at(const Field& f, Site s, int mu) {
        return (s.p ? f.l[1] : f.l[0]) + (size_t)(18 * mu) * f.Vh + (s.lex >> 1);
    }
    // entry i of column j of the matrix: U, its transpose (T), complex conjugate (C) or both
    template <bool T, bool C>
    static __device__ __forceinline__ Vec3<R> column(const Field& f, Site s, int mu, int j) {
        const uint4* m = at(f, s, mu);
        Vec3<R> o;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint4 w = __ldg(m + (size_t)(T ? 3 * j + i : 3 * i + j) * f.Vh);
            const R re = ((R)(int)w.y << 32) + (int)w.x, im = ((R)(int)w.w << 32) + (int)w.z;
            o.v[2 * i] = re >> 2;
            o.v[2 * i + 1] = C ? -(im >> 2) : im >> 2;
        }
        return o;
    }
    template <bool T, bool C>
    static __device__ __noinline__ Vec3<R> mul(const uint4* m, int Vh, Vec3<R> v) {
        int h0[6], h1[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) fx::digits(v.v[i], h0[i], h1[i]);
        Vec3<R> o;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            int u0[6], u1[6], n0[3], n1[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const uint4 w = __ldg(m + (size_t)(T ? 3 * j + i : 3 * i + j) * Vh);
                u0[2 * j] = (int)w.x;
                u1[2 * j] = (int)w.y;
                u0[2 * j + 1] = C ? -(int)w.z : (int)w.z;
                u1[2 * j + 1] = C ? -(int)w.w : (int)w.w;
                n0[j] = C ? (int)w.z : -(int)w.z;
                n1[j] = C ? (int)w.w : -(int)w.w;
            }
            long long re, im;
            fx::row_mul(u0, u1, n0, n1, h0, h1, re, im);
            o.v[2 * i] = re * 8;
            o.v[2 * i + 1] = im * 8;
        }
        return o;
    }
    template <bool T, bool C>
    static __device__ __forceinline__ Vec3<R> mul(const Field& f, Site s, int mu, Vec3<R> v) {
        return mul<T, C>(at(f, s, mu), f.Vh, v);
    }
    static __device__ __forceinline__ double real(R v) { return (double)v * (1.0 / 576460752303423488.0); }   // 2^-59
};

template <> struct Links<false> {
    typedef double R;
    static __device__ __forceinline__ const double* at(const Field& f, Site s, int mu) {
        return f.U + ((size_t)mu * f.V + s.lex) * 18;
    }
    template <bool T, bool C>
    static __device__ __forceinline__ Vec3<R> column(const Field& f, Site s, int mu, int j) {
        const double* m = at(f, s, mu);
        Vec3<R> o;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int e = 2 * (T ? 3 * j + i : 3 * i + j);
            o.v[2 * i] = m[e];
            o.v[2 * i + 1] = C ? -m[e + 1] : m[e + 1];
        }
        return o;
    }
    template <bool T, bool C>
    static __device__ __noinline__ Vec3<R> mul(const double* m, Vec3<R> v) {
        Vec3<R> o;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            double re = 0.0, im = 0.0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int e = 2 * (T ? 3 * j + i : 3 * i + j);
                const double a = m[e], b = C ? -m[e + 1] : m[e + 1];
                re = fma(-b, v.v[2 * j + 1], fma(a, v.v[2 * j], re));
                im = fma(b, v.v[2 * j], fma(a, v.v[2 * j + 1], im));
            }
            o.v[2 * i] = re;
            o.v[2 * i + 1] = im;
        }
        return o;
    }
    template <bool T, bool C>
    static __device__ __forceinline__ Vec3<R> mul(const Field& f, Site s, int mu, Vec3<R> v) {
        return mul<T, C>(at(f, s, mu), v);
    }
    static __device__ __forceinline__ double real(R v) { return v; }
};

// Site at coordinates c shifted by a mu-hat + b nu-hat (a, b in -1..1), periodic.
__device__ __forceinline__ Site shifted(const Geom& g, const Coord& c, int mu, int a, int nu, int b) {
    int d[4] = {c.x, c.y, c.z, c.t};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int s = (i == mu ? a : 0) + (i == nu ? b : 0);
        d[i] += s;
        if (d[i] < 0) d[i] += g.L[i];
        if (d[i] >= g.L[i]) d[i] -= g.L[i];
    }
    return {d[0] + g.L[0] * (d[1] + g.L[1] * (d[2] + g.L[2] * d[3])), (d[0] + d[1] + d[2] + d[3]) & 1};
}

// Q - Q^+ of plane (mu, nu) from two products of three links each. The leaves L1..L4 enter only through their
// anti-Hermitian parts, so L2 may be replaced by -L2^+, which ends with U_nu(x)^+ as L1 does, and L4 by -L4^+,
// which ends with U_nu(x - nu) as L3 does:
//   L1 - L2^+ = [U_mu(x) U_nu(x+mu) U_mu(x+nu)^+ - U_mu(x-mu)^+ U_nu(x-mu) U_mu(x-mu+nu)] U_nu(x)^+
//   L3 - L4^+ = [U_mu(x-mu)^+ U_nu(x-mu-nu)^+ U_mu(x-mu-nu) - U_mu(x) U_nu(x+mu-nu)^+ U_mu(x-nu)^+] U_nu(x-nu)
// (10 matrix products instead of 12). Writes the 9 reals of F before the trace is taken out: diagonal, then the
// complex elements (0,1), (0,2), (1,2).
template <bool FIXED>
__device__ void plane_field(const Geom& g, const Field& f, const Coord& c, int mu, int nu, double (&F)[9]) {
    typedef Links<FIXED> L;
    typedef typename L::R R;
    const Site x = shifted(g, c, mu, 0, nu, 0), xm = shifted(g, c, mu, -1, nu, 0), xn = shifted(g, c, mu, 0, nu, -1);
    R q[3][6];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        Vec3<R> X[3];   // columns
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            Vec3<R> a, b;
            if (half == 0) {
                const Site pn = shifted(g, c, mu, 0, nu, 1), pm = shifted(g, c, mu, 1, nu, 0);
                const Site mp = shifted(g, c, mu, -1, nu, 1);
                a = L::template column<true, true>(f, pn, mu, j);
                a = L::template mul<false, false>(f, pm, nu, a);
                a = L::template mul<false, false>(f, x, mu, a);
                b = L::template column<false, false>(f, mp, mu, j);
                b = L::template mul<false, false>(f, xm, nu, b);
                b = L::template mul<true, true>(f, xm, mu, b);
            } else {
                const Site mm = shifted(g, c, mu, -1, nu, -1), pm = shifted(g, c, mu, 1, nu, -1);
                a = L::template column<false, false>(f, mm, mu, j);
                a = L::template mul<true, true>(f, mm, nu, a);
                a = L::template mul<true, true>(f, xm, mu, a);
                b = L::template column<true, true>(f, xn, mu, j);
                b = L::template mul<true, true>(f, pm, nu, b);
                b = L::template mul<false, false>(f, x, mu, b);
            }
#pragma unroll
            for (int e = 0; e < 6; ++e) X[j].v[e] = a.v[e] - b.v[e];
        }
        // row i of X W: the vector X_i. through W^T
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Vec3<R> r;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                r.v[2 * j] = X[j].v[2 * i];
                r.v[2 * j + 1] = X[j].v[2 * i + 1];
            }
            r = half == 0 ? L::template mul<false, true>(f, x, nu, r) : L::template mul<true, false>(f, xn, nu, r);
#pragma unroll
            for (int e = 0; e < 6; ++e) q[i][e] = half == 0 ? r.v[e] : q[i][e] + r.v[e];
        }
    }
    // F = (Q - Q^+) / (8 i): (re, im) -> (im, -re) / 8
#pragma unroll
    for (int i = 0; i < 3; ++i) F[i] = 0.25 * L::real(q[i][2 * i + 1]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = k < 2 ? 0 : 1, j = k < 1 ? 1 : 2;
        F[3 + 2 * k] = 0.125 * L::real(q[i][2 * j + 1] + q[j][2 * i + 1]);
        F[4 + 2 * k] = -0.125 * L::real(q[i][2 * j] - q[j][2 * i]);
    }
}

// Packed block c of site h: 36 reals and 4 zeros as 20 units.
__device__ __forceinline__ void store_chiral(uint4* dst, int Vh, int h, int c, const double (&s)[36]) {
#pragma unroll
    for (int u = 0; u < 20; ++u) {
        const double v[2] = {u < 18 ? s[2 * u < 36 ? 2 * u : 0] : 0.0, u < 18 ? s[2 * u + 1 < 36 ? 2 * u + 1 : 0] : 0.0};
        dst[(size_t)(20 * c + u) * Vh + h] = Unit<double>::put(v);
    }
}

// Largest real of F below which a plane's products are formed in FP64 arithmetic also for SU(3) links. FP64 arithmetic
// holds F to 2e-16 of its largest element whatever its size (the imaginary parts of near-unit links are products with
// one small factor), fixed point to 2e-18 absolute times a few: 2e-17 of F at 0.3, 6e-17 at 0.1, 2e-16 at 0.03, 6e-15
// at 1e-3 (rms over random links).
constexpr double WEAK_FIELD = 0.0625;

// One block takes 32 sites of one parity (blockIdx.y): each of its six warps
// forms the field strength of one plane, then warps 0 and 1 assemble and
// invert one chiral block each. Bound: in FP64 arithmetic the products (6480
// multiply-adds per site) keep the FP64 pipe busy; in fixed point they take the
// integer multiplier a quarter of that time, and the inverses (~1000 FP64
// operations) are half of the rest. Measured at 24^3 x 48: 3.6 ms (3.3 without
// the weak planes in FP64 arithmetic), against 53.7 ms with one thread per site and 12 x 12 blocks in local memory.
template <bool FIXED>
__global__ void __launch_bounds__(192) k_clover_build(Geom g, Field f, double ck, uint4* fwd_e, uint4* fwd_o,
                                                      uint4* inv_e, uint4* inv_o, int* singular) {
    __shared__ double F[6][9][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, p = blockIdx.y;
    const int h = blockIdx.x * 32 + lane;
    const bool ok = h < g.Vh;
    if (ok) {
        const int mu = warp < 3 ? 0 : warp < 5 ? 1 : 2;
        const int nu = warp < 3 ? warp + 1 : warp < 5 ? warp - 1 : 3;
        double t[9];
        const Coord c = coord_of(g, p, h);
        plane_field<FIXED>(g, f, c, mu, nu, t);
        if (FIXED) {   // a weak field is smaller than the products it is left over from: FP64 arithmetic
            double most = 0.0;
            for (int i = 0; i < 9; ++i) most = fmax(most, fabs(t[i]));
            if (most < WEAK_FIELD) plane_field<false>(g, f, c, mu, nu, t);
        }
        const double tr = (t[0] + t[1] + t[2]) / 3.0;
        for (int i = 0; i < 9; ++i) F[warp][i][lane] = i < 3 ? t[i] - tr : t[i];
    }
    __syncthreads();
    if (!ok || warp > 1) return;
    // planes (0,1) (0,2) (0,3) (1,2) (1,3) (2,3) are warps 0..5
    const double sg = warp == 0 ? -1.0 : 1.0, hk = 0.5 * ck;
    double gx[9], gy[9], gz[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        gx[i] = hk * fma(sg, F[2][i][lane], F[3][i][lane]);
        gy[i] = hk * fma(sg, F[4][i][lane], -F[1][i][lane]);
        gz[i] = hk * fma(sg, F[5][i][lane], F[0][i][lane]);
    }
    double s[36];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        s[i] = gz[i];
        s[3 + i] = -gz[i];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // (a, b) element of G: diagonal real, upper triangle stored, lower its conjugate
            auto el = [&](const double (&m)[9], double& re, double& im) {
                const int lo = i < j ? i : j, hi = i < j ? j : i, q = 3 + 2 * (lo + hi - 1);
                re = i == j ? m[i] : m[i == j ? 0 : q];
                im = i == j ? 0.0 : i < j ? m[i == j ? 0 : q + 1] : -m[i == j ? 0 : q + 1];
            };
            double xr, xi, yr, yi, zr, zi;
            el(gx, xr, xi);
            el(gy, yr, yi);
            el(gz, zr, zi);
            if (i < j) {
                s[herm6::tri(i, j)] = zr;
                s[herm6::tri(i, j) + 1] = zi;
                s[herm6::tri(3 + i, 3 + j)] = -zr;
                s[herm6::tri(3 + i, 3 + j) + 1] = -zi;
            }
            s[herm6::tri(i, 3 + j)] = xr + yi;       // G_x - i G_y
            s[herm6::tri(i, 3 + j) + 1] = xi - yr;
        }
    }
    store_chiral(p == 0 ? fwd_e : fwd_o, g.Vh, h, warp, s);
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] += 0.5;
    double r[36];
#pragma unroll
    for (int i = 0; i < 36; ++i) r[i] = s[i];
    if (!herm6::sweep_inverse(r)) {
        double in[36], out[36];
        for (int i = 0; i < 36; ++i) in[i] = s[i];
        if (!herm6::invert_pivoted(in, out)) atomicExch(singular, 1);
        else
            for (int i = 0; i < 36; ++i) r[i] = out[i];
    }
#pragma unroll
    for (int i = 0; i < 36; ++i) r[i] *= 0.25;
    store_chiral(p == 0 ? inv_e : inv_o, g.Vh, h, warp, r);
}

}  // namespace

// (Re)build the FP64 clover blocks of the handle's gauge field; lower-precision
// copies are dropped and rebuilt on first use.
int clover_build(wd_handle* h) {
    const size_t bytes = (size_t)h->g.Vh * 40 * 16;
    // blocks that are there are rewritten in place, the lower precisions on their next use: work on any stream that
    // still reads them has to be done
    if (h->clov64[0][0]) WD_CUDA(h, cudaDeviceSynchronize());
    uint4* b[4];
    const char* names[4] = {"clov.fwd64.e", "clov.fwd64.o", "clov.inv64.e", "clov.inv64.o"};
    for (int i = 0; i < 4; ++i) {
        b[i] = (uint4*)workspace(h, names[i], bytes);
        if (!b[i]) return fail(h, WD_ERR_CUDA, "out of device memory (clover blocks)");
    }
    int* sing = (int*)workspace(h, "clov.singular", sizeof(int));
    if (!sing) return fail(h, WD_ERR_CUDA, "out of device memory");
    WD_CUDA(h, cudaMemset(sing, 0, sizeof(int)));
    Field f{h->U64, {nullptr, nullptr}, 2LL * h->g.Vh, h->g.Vh};
    if (h->fixed64) {   // SU(3) links: the products in fixed point, from the gathered FP64 links
        const int rc = ensure_links(h, WD_FP64, 18, &f.l[0], &f.l[1]);
        if (rc != WD_OK) return rc;
    }
    const dim3 grid((h->g.Vh + 31) / 32, 2);
    const double ck = h->csw * h->kappa;
    if (h->fixed64) k_clover_build<true><<<grid, 192>>>(h->g, f, ck, b[0], b[1], b[2], b[3], sing);
    else k_clover_build<false><<<grid, 192>>>(h->g, f, ck, b[0], b[1], b[2], b[3], sing);
    WD_CUDA(h, cudaGetLastError());
    int hs = 0;
    WD_CUDA(h, cudaMemcpy(&hs, sing, sizeof(int), cudaMemcpyDeviceToHost));
    if (hs) return fail(h, WD_ERR_INVALID_ARG, "wd_set_clover: a clover block is singular");
    for (int k = 0; k < 2; ++k)
        for (int p = 0; p < 4; ++p) h->clov[k][p][0] = h->clov[k][p][1] = nullptr;
    for (int p = 0; p < 2; ++p) {
        h->clov64[1][p] = b[p];
        h->clov64[0][p] = b[2 + p];
    }
    h->gen += 1;
    return WD_OK;
}

// Clover blocks of kind 0 (C^{-1}) or 1 (C - 1) in precision prec (chiral packing)
// for both parities; null pointers when the handle has no clover term.
int ensure_clover(wd_handle* h, int prec, int kind, const uint4** even, const uint4** odd) {
    *even = *odd = nullptr;
    if (!h->have_clover) return WD_OK;
    for (int p = 0; p < 2; ++p) {
        if (prec == WD_FP64) {
            h->clov[kind][prec][p] = h->clov64[kind][p];
        } else if (!h->clov[kind][prec][p]) {
            const size_t units = 80 / (prec == WD_FP32 ? 4 : 2 * 4);
            const std::string name = "clov.k" + std::to_string(kind) + ".p" + std::to_string(prec) + "." +
                                     std::to_string(p);
            uint4* dst = (uint4*)workspace(h, name, (size_t)h->g.Vh * units * 16);
            if (!dst) return fail(h, WD_ERR_CUDA, "out of device memory (clover blocks)");
            const uint4* src = h->clov64[kind][p];
            cudaError_t e = by_prec(prec, [&](auto tag) {
                typedef typename decltype(tag)::type T;
                return Ops<T>::chiral_from64(h->g.Vh, src, dst, nullptr);
            });
            WD_CUDA(h, e);
            WD_CUDA(h, cudaDeviceSynchronize());
            h->clov[kind][prec][p] = dst;
        }
    }
    *even = h->clov[kind][prec][0];
    *odd = h->clov[kind][prec][1];
    return WD_OK;
}

}  // namespace wd

using namespace wd;

extern "C" int wd_set_clover(wd_handle* h, double csw) {
    if (!h) return WD_ERR_INVALID_ARG;
    if (!std::isfinite(csw)) return fail(h, WD_ERR_INVALID_ARG, "wd_set_clover: c_sw must be finite");
    if (!h->have_gauge) return fail(h, WD_ERR_NO_GAUGE, "wd_set_clover: wd_set_gauge has not been called");
    if (h->g.part && csw != 0.0) return fail(h, WD_ERR_INVALID_ARG, "wd_set_clover: a split lattice (wd_dd_set_partition) has only the wd_dd_* operators");
    if (csw == 0.0) {
        h->have_clover = false;
        h->csw = 0.0;
        for (int k = 0; k < 2; ++k)
            for (int p = 0; p < 4; ++p) h->clov[k][p][0] = h->clov[k][p][1] = nullptr;
        h->gen += 1;
        return WD_OK;
    }
    h->csw = csw;
    int rc = clover_build(h);
    if (rc != WD_OK) {
        h->have_clover = false;
        return rc;
    }
    h->have_clover = true;
    return WD_OK;
}

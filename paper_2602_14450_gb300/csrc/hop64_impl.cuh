// The FP64 hop on the integer pipes (fixed64.cuh): the same operation as
// hop_kernel<double, 18> (hop_impl.cuh) for SU(3) links held as fixed-point
// digits, one site per thread.
#pragma once

#include "fixed64.cuh"
#include "hop_impl.cuh"

namespace wd {

#define RE(s, c) (2 * (3 * (s) + (c)))
#define IM(s, c) (2 * (3 * (s) + (c)) + 1)

// The hop of one site in FP64 arithmetic from the fixed-point links, direction by direction: taken by sites with
// a neighbour outside the fixed-point range (not finite, or with reals near the ends of the exponent range).
static __device__ __noinline__ void hop64_site(const HopParams& P, const uint4* vin, int h, double* out) {
    const Geom& g = P.g;
    int nbr[8];
    const unsigned wm = site_neighbours(g, P.parity, h, nbr);
    double acc[24];
    for (int i = 0; i < 24; ++i) acc[i] = 0.0;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        if (((wm >> d) & 1u) && ((g.part >> mu) & 1u)) continue;   // leaves the sub-lattice
        double nb[24], hs[12], chi[12];
        uint4 u[9];
        load_spinor<double>(vin, g.Vh, nbr[d], nb);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const uint4 w = __ldg(P.links + (size_t)(9 * d + k) * g.Vh + h);
            const double v[2] = {fx::link_value((int)w.x, (int)w.y), fx::link_value((int)w.z, (int)w.w)};
            u[k] = Unit<double>::put(v);
        }
        project<double>(mu, fwd, nb, hs);
        link_mul<double, 18>(u, 0, hs, chi);
        const double f = (mu == 3 ? 2.0 : 1.0) * ((((wm >> d) & 1u) && g.bc[mu] < 0) ? -1.0 : 1.0);
        reconstruct<double>(mu, fwd, f, chi, acc);
    }
    for (int i = 0; i < 24; ++i) out[i] = acc[i];
}

// acc += rebuilt four-spinor of x = U h (column k, row c, (re, im) at 6 k + 2 c), as reconstruct().
__device__ __forceinline__ void rebuild_fixed(int mu, bool fwd, const long long (&x)[12], long long (&acc)[24]) {
    auto add = [&](int i, bool plus, long long v) { acc[i] = plus ? acc[i] + v : acc[i] - v; };
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long x0r = x[2 * c], x0i = x[2 * c + 1], x1r = x[6 + 2 * c], x1i = x[6 + 2 * c + 1];
        if (mu == 3) {
            const int a0 = fwd ? 2 : 0, a1 = fwd ? 3 : 1;
            acc[RE(a0, c)] += x0r + x0r;
            acc[IM(a0, c)] += x0i + x0i;
            acc[RE(a1, c)] += x1r + x1r;
            acc[IM(a1, c)] += x1i + x1i;
            continue;
        }
        acc[RE(0, c)] += x0r;
        acc[IM(0, c)] += x0i;
        acc[RE(1, c)] += x1r;
        acc[IM(1, c)] += x1i;
        if (mu == 0) {          // comp2 = -s i chi1, comp3 = -s i chi0
            add(RE(2, c), fwd, x1i);
            add(IM(2, c), !fwd, x1r);
            add(RE(3, c), fwd, x0i);
            add(IM(3, c), !fwd, x0r);
        } else if (mu == 1) {   // comp2 = -s chi1, comp3 = s chi0
            add(RE(2, c), !fwd, x1r);
            add(IM(2, c), !fwd, x1i);
            add(RE(3, c), fwd, x0r);
            add(IM(3, c), fwd, x0i);
        } else {                // comp2 = -s i chi0, comp3 = s i chi1
            add(RE(2, c), fwd, x0i);
            add(IM(2, c), !fwd, x0r);
            add(RE(3, c), !fwd, x1i);
            add(IM(3, c), fwd, x1r);
        }
    }
}

constexpr int HOP64_THREADS = 128;
// Resident blocks per SM: 4 (128 registers). 3 (168 registers) is 2% faster at 32^3 x 64 (425 against 435 us), but at
// 16^3 x 32 it leaves 56 of the 512 blocks to a second wave.
constexpr int HOP64_BLOCKS = 4;

// Bounds: a warp issues about 7500 instructions per 32 sites, 1728 of them
// wide integer multiply-adds, which occupy the multiplier pipe 4.4-5.7 cycles
// each (measured; 2.1 for other integer multiply-adds): ~0.3 of the 0.425 ms
// at 32^3 x 64; the 1.6 GB of links and vectors take 0.24 ms. The same hop in
// FP64 arithmetic (hop_kernel<double, 18>) takes 1.437 ms, all of it FP64 pipe.
//
// The eight directions run as one loop body rather than unrolled: unrolled,
// the straight-line code ran at the rate of the instruction cache (770 us).
// The spin structure is selected at run time: the partner spins of the
// projection by the load addresses, the factor i by a selection of words,
// signs by masks, and the rebuild by a branch that is the same for the whole
// warp. The links arrive through a two-slot ring in shared memory filled by
// cp.async one direction ahead, which holds no registers (without it: 472 us,
// a third of the stalls waiting for links).
template <int EPI, int RED, bool MAT>
__global__ void __launch_bounds__(HOP64_THREADS, HOP64_BLOCKS) hop64_kernel(const HopParams P) {
    [[maybe_unused]] constexpr unsigned wd_tl_tag = RED;   // timeline records: the reduction
    pdl_begin();
    constexpr int NS = RedSums<RED>::N;
    // this thread's neighbours and a two-slot ring of its links, copied one direction ahead (cp.async); each thread
    // reads only what it wrote or copied itself
    __shared__ int nbs[8][HOP64_THREADS];
    __shared__ uint4 ring[2][9][HOP64_THREADS];
    const Slice sl = slice_of(P.nrhs);
    if (guarded(P.guard ? P.guard + sl.rhs : nullptr, P.guard_kind)) return;
    const long long ro = (long long)sl.rhs * P.vs;     // this right-hand side's vectors
    const uint4* __restrict__ vin = P.in + ro;
    uint4* vout = P.out + ro;
    const uint4* vy = P.y ? P.y + ro : nullptr;
    const uint4* vz = P.z ? P.z + ro : nullptr;
    const uint4* vrs = P.rstar ? P.rstar + ro : nullptr;
    const Geom& g = P.g;
    const int Vh = g.Vh;
    double part[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) part[k] = 0;

    for (int h = sl.b * blockDim.x + threadIdx.x; h < Vh; h += sl.nb * blockDim.x) {
        unsigned neg;          // directions whose hop carries a boundary phase -1
        {
            int nbr[8];
            neg = site_neighbours(g, P.parity, h, nbr);   // those that wrap around
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                // -1: a hop that leaves the sub-lattice of a split direction has no neighbour here
                nbs[d][threadIdx.x] = ((neg >> d) & 1u) && ((g.part >> (d >> 1)) & 1u) ? -1 : nbr[d];
                if (g.bc[d >> 1] > 0) neg &= ~(1u << d);
            }
        }
        auto copy_links = [&](int d) {
            const uint4* lp = P.links + (size_t)(9 * d) * Vh + h;
#pragma unroll
            for (int k = 0; k < 9; ++k) cp_async16(&ring[d & 1][k][threadIdx.x], lp + (size_t)k * Vh);
            cp_async_commit();
        };
        copy_links(0);
        long long acc[24];
#pragma unroll
        for (int i = 0; i < 24; ++i) acc[i] = 0;
        int E = 0;             // exponent of acc; 0 while every neighbour so far was zero
        bool bad = false;
#pragma unroll 1
        for (int d = 0; d < 8; ++d) {
            const int mu = d >> 1, hn = nbs[d][threadIdx.x];
            if (hn < 0) {
                if (d + 1 < 8) copy_links(d + 1);
                else cp_async_commit();
                cp_async_wait<1>();          // the next copy reuses the slot of the one before this
                continue;
            }
            // upper spins p (of the t hops: the pair the projector keeps) and their partners q
            const uint4* np = vin + hn;
            const uint4* pp = np + (size_t)(d == 6 ? 6 : 0) * Vh;
            uint4 p[6], q[6];
#pragma unroll
            for (int u = 0; u < 6; ++u) p[u] = __ldg(pp + (size_t)u * Vh);
            if (mu < 3) {
                const uint4* q0 = np + (size_t)(mu == 2 ? 6 : 9) * Vh;
                const uint4* q1 = np + (size_t)(mu == 2 ? 9 : 6) * Vh;
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    q[u] = __ldg(q0 + (size_t)u * Vh);
                    q[3 + u] = __ldg(q1 + (size_t)u * Vh);
                }
            } else {
#pragma unroll
                for (int u = 0; u < 6; ++u) q[u] = make_uint4(0u, 0u, 0u, 0u);
            }
            if (d + 1 < 8) copy_links(d + 1);
            else cp_async_commit();          // empty group: the wait below counts the same way
            unsigned top = 0;
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                top = max(top, max(p[u].y & 0x7FFFFFFFu, p[u].w & 0x7FFFFFFFu));
                top = max(top, max(q[u].y & 0x7FFFFFFFu, q[u].w & 0x7FFFFFFFu));
            }
            const int En = (int)(top >> 20);
            if (En < fx::E_MIN || En > fx::E_MAX) {
                unsigned any = top;
#pragma unroll
                for (int u = 0; u < 6; ++u) any |= p[u].x | p[u].z | q[u].x | q[u].z;
                if (any != 0) bad = true;    // a zero half spinor adds nothing
                cp_async_wait<1>();          // the next copy reuses the slot of the one before this
                continue;
            }
            if (En > E) {
                // one binade above, which most later neighbours stay below: fewer shifts (913 -> 896 us for D_W)
                const int Ek = min(En + 1, fx::E_MAX);
                if (E) {
                    const int sh = min(Ek - E, 63);
#pragma unroll
                    for (int i = 0; i < 24; ++i) acc[i] >>= sh;
                }
                E = Ek;
            }
            if ((neg >> d) & 1u) {
#pragma unroll
                for (int u = 0; u < 6; ++u) {
                    p[u].y ^= 0x80000000u;
                    p[u].w ^= 0x80000000u;
                    q[u].y ^= 0x80000000u;
                    q[u].w ^= 0x80000000u;
                }
            }
            // half spinor, the projections of project() (hop_impl.cuh): column k = 0, 1 is p_k + f_k q_k with
            // f = s i, s i (mu = 0); s, -s (1); s i, -s i (2); s = +1 forward, -1 backward
            int h0[12], h1[12];
            const bool rot = mu != 1;
            const int s = (d & 1) ? -1 : 0, s1 = mu == 0 ? s : ~s;
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                const int mi = u < 3 ? s : s1, mr = rot ? ~mi : mi;
                const fx::Fixed pr = fx::fixed(p[u].y, p[u].x, E), pi = fx::fixed(p[u].w, p[u].z, E);
                const fx::Fixed qr = fx::fixed(rot ? q[u].w : q[u].y, rot ? q[u].z : q[u].x, E);
                const fx::Fixed qi = fx::fixed(rot ? q[u].y : q[u].w, rot ? q[u].x : q[u].z, E);
                fx::digits(fx::sum(pr, fx::signed_by(qr, mr)), h0[2 * u], h1[2 * u]);
                fx::digits(fx::sum(pi, fx::signed_by(qi, mi)), h0[2 * u + 1], h1[2 * u + 1]);
            }
            cp_async_wait<1>();
            long long x[12];   // U h: column k, row c, (re, im) at 6 k + 2 c
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                int l0[6], l1[6], n0[3], n1[3];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const uint4 w = ring[d & 1][3 * c + b][threadIdx.x];
                    l0[2 * b] = (int)w.x;
                    l1[2 * b] = (int)w.y;
                    l0[2 * b + 1] = (int)w.z;
                    l1[2 * b + 1] = (int)w.w;
                    n0[b] = -(int)w.z;
                    n1[b] = -(int)w.w;
                }
                fx::row_mul(l0, l1, n0, n1, h0, h1, x[2 * c], x[2 * c + 1]);
                fx::row_mul(l0, l1, n0, n1, h0 + 6, h1 + 6, x[6 + 2 * c], x[6 + 2 * c + 1]);
            }
            switch (d) {
            case 0: rebuild_fixed(0, true, x, acc); break;
            case 1: rebuild_fixed(0, false, x, acc); break;
            case 2: rebuild_fixed(1, true, x, acc); break;
            case 3: rebuild_fixed(1, false, x, acc); break;
            case 4: rebuild_fixed(2, true, x, acc); break;
            case 5: rebuild_fixed(2, false, x, acc); break;
            case 6: rebuild_fixed(3, true, x, acc); break;
            default: rebuild_fixed(3, false, x, acc); break;
            }
        }
        cp_async_wait<0>();      // a site left early may have a copy in flight
        double o[24];
        if (bad) {
            double t[24];
            hop64_site(P, vin, h, t);
            for (int i = 0; i < 24; ++i) o[i] = t[i];
        } else {
#pragma unroll
            for (int i = 0; i < 24; ++i) o[i] = fx::to_double(acc[i], E);
        }
        hop_epilogue<double, EPI, RED, MAT>(P, vout, vy, vz, vrs, h, o, part, false);
    }
    if constexpr (RED != RED_NONE) grid_reduce<NS, RedStage<RED>::HINT>(part, P.rc, sl);
}

#undef RE
#undef IM

}  // namespace wd

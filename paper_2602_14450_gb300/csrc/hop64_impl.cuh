// The FP64 hop on the integer pipes (fixed64.cuh): the same operation as
// hop_kernel<double, 18> (hop_impl.cuh) for SU(3) links held as fixed-point
// digits, one site per thread. Sites where fixed point could be less exact than
// FP64 arithmetic, in any of their 24 reals, are done in FP64 arithmetic.
#pragma once

#include "fixed64.cuh"
#include "hop_impl.cuh"

namespace wd {

#define RE(s, c) (2 * (3 * (s) + (c)))
#define IM(s, c) (2 * (3 * (s) + (c)) + 1)

__device__ __forceinline__ double negated(double x, bool n) { return n ? -x : x; }

// The hop of the sites h of the lanes with `take` set, in FP64 arithmetic from the FP64 links (host layout): sites
// with a neighbour outside the fixed-point range (not finite, or with reals near the ends of the exponent range) and
// those with a real that fails the size test of hop64_kernel. Called by whole warps. Eight lanes share a site, one
// direction each, and the shares are added in the order of hop_kernel: an FP64 instruction occupies the pipe 64 cycles whatever the
// number of lanes, so one lane for a site made a launch with a single such site 50 us longer (16^3 x 32, FP64 solve:
// 68.6 ms).
static __device__ __noinline__ void hop64_sites(const HopParams& P, const uint4* vin, int h, bool take, double* out) {
    constexpr unsigned ALL = 0xFFFFFFFFu;
    const Geom& g = P.g;
    const int lane = threadIdx.x & 31, d = lane & 7, mu = d >> 1;
    const bool back = d & 1, rot = mu == 0 || mu == 2;
    const size_t V = 2 * (size_t)g.Vh;
    for (unsigned todo = __ballot_sync(ALL, take); todo != 0;) {
        int src = -1, mine = -1;   // the lane whose site this group of eight takes; the group that takes this lane's site
        for (int k = 0; k < 4 && todo != 0; ++k, todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            if (k == lane >> 3) src = l;
            if (l == lane) mine = k;
        }
        const int hs = __shfl_sync(ALL, h, src < 0 ? lane : src);
        double x[12];              // U h of this lane's direction: column k, row c, (re, im) at 6 k + 2 c
#pragma unroll
        for (int i = 0; i < 12; ++i) x[i] = 0.0;
        bool wrap;
        const int hn = neighbour(g, hs, coord_of(g, P.parity, hs), d, &wrap);
        if (src >= 0 && !(wrap && ((g.part >> mu) & 1u))) {
            const uint4* np = vin + hn;
            const uint4* pp = np + (size_t)(d == 6 ? 6 : 0) * g.Vh;
            const uint4* qp[2] = {np + (size_t)(mu == 2 ? 6 : 9) * g.Vh, np + (size_t)(mu == 2 ? 9 : 6) * g.Vh};
            double hv[12];
#pragma unroll
            for (int k = 0; k < 2; ++k) {   // column k of the half spinor: p_k + f q_k, as in hop64_kernel
                const bool neg = back != (k == 1 && mu != 0);
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const uint4 p = __ldg(pp + (size_t)(3 * k + b) * g.Vh);
                    const uint4 q = mu < 3 ? __ldg(qp[k] + (size_t)b * g.Vh) : make_uint4(0u, 0u, 0u, 0u);
                    const double qr = Unit<double>::get(q, 0), qi = Unit<double>::get(q, 1);
                    hv[6 * k + 2 * b] = Unit<double>::get(p, 0) + negated(rot ? qi : qr, neg != rot);
                    hv[6 * k + 2 * b + 1] = Unit<double>::get(p, 1) + negated(rot ? qr : qi, neg);
                }
            }
            const size_t from = lex_of(g, back ? 1 - P.parity : P.parity, back ? hn : hs);
            const double2* lp = reinterpret_cast<const double2*>(P.U64 + (mu * V + from) * 18);
            const bool minus = wrap && g.bc[mu] < 0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                double m[6];
#pragma unroll
                for (int b = 0; b < 3; ++b) {   // U, or U^+ backwards
                    const double2 w = __ldg(lp + (back ? 3 * b + c : 3 * c + b));
                    m[2 * b] = w.x;
                    m[2 * b + 1] = negated(w.y, back);
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const double* v = hv + 6 * k;
                    double re = m[0] * v[0], im = m[0] * v[1];
                    re = fma(-m[1], v[1], re);
                    im = fma(m[1], v[0], im);
#pragma unroll
                    for (int b = 1; b < 3; ++b) {
                        re = fma(-m[2 * b + 1], v[2 * b + 1], fma(m[2 * b], v[2 * b], re));
                        im = fma(m[2 * b + 1], v[2 * b], fma(m[2 * b], v[2 * b + 1], im));
                    }
                    x[6 * k + 2 * c] = negated(re, minus);
                    x[6 * k + 2 * c + 1] = negated(im, minus);
                }
            }
        }
        // the direction's share of each real (rebuild_fixed), and this lane's sums over the eight lanes of its group
        const bool n2 = mu < 3 && !back, n3 = mu == 0 ? !back : mu < 3 && back;
        double o[24];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double x0r = x[2 * c], x0i = x[2 * c + 1], x1r = x[6 + 2 * c], x1i = x[6 + 2 * c + 1];
            const double ar = mu < 2 ? x1r : x0r, ai = mu < 2 ? x1i : x0i, br = mu < 2 ? x0r : x1r, bi = mu < 2 ? x0i : x1i;
            o[RE(0, c)] = d == 6 ? 0.0 : x0r;
            o[IM(0, c)] = d == 6 ? 0.0 : x0i;
            o[RE(1, c)] = d == 6 ? 0.0 : x1r;
            o[IM(1, c)] = d == 6 ? 0.0 : x1i;
            o[RE(2, c)] = d == 7 ? 0.0 : negated(rot ? ai : ar, n2 != rot);
            o[IM(2, c)] = d == 7 ? 0.0 : negated(rot ? ar : ai, n2);
            o[RE(3, c)] = d == 7 ? 0.0 : negated(rot ? bi : br, n3 != rot);
            o[IM(3, c)] = d == 7 ? 0.0 : negated(rot ? br : bi, n3);
        }
#pragma unroll
        for (int i = 0; i < 24; ++i) {
            double sum = 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const double v = __shfl_sync(ALL, o[i], 8 * (mine < 0 ? 0 : mine) + k);
                sum = k < 6 ? sum + v : fma(2.0, v, sum);   // the t hops count twice
            }
            if (mine >= 0) out[i] = sum;
        }
    }
}

// The sizes of three integers by their upper bytes, one in each of the lower three bytes (negative ones rounded down).
__device__ __forceinline__ unsigned sizes(int x0, int x1, int x2) {
    const unsigned p = __byte_perm(__byte_perm(x0, x1, 0x0073), x2, 0x0710);
    unsigned neg;   // the sign of each byte in all its bits
    asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(neg) : "r"(p));
    return (p ^ neg) & 0xFFFFFFu;
}

// acc += rebuilt four-spinor of x = U h (column k, row c, (re, im) at 6 k + 2 c), as reconstruct(); tot += the sizes
// z of the products in x (column k, row c at 3 k + c; real part low, imaginary part high), spin s, colour c at 3 s + c.
__device__ __forceinline__ void rebuild_fixed(int mu, bool fwd, const long long (&x)[12], const unsigned (&z)[6],
                                              long long (&acc)[24], unsigned (&tot)[12]) {
    auto add = [&](int i, bool plus, long long v) { acc[i] = plus ? acc[i] + v : acc[i] - v; };
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long x0r = x[2 * c], x0i = x[2 * c + 1], x1r = x[6 + 2 * c], x1i = x[6 + 2 * c + 1];
        const unsigned z0 = z[c], z1 = z[3 + c];
        if (mu == 3) {
            const int a0 = fwd ? 2 : 0, a1 = fwd ? 3 : 1;
            acc[RE(a0, c)] += x0r + x0r;
            acc[IM(a0, c)] += x0i + x0i;
            acc[RE(a1, c)] += x1r + x1r;
            acc[IM(a1, c)] += x1i + x1i;
            tot[3 * a0 + c] += 2 * z0;
            tot[3 * a1 + c] += 2 * z1;
            continue;
        }
        acc[RE(0, c)] += x0r;
        acc[IM(0, c)] += x0i;
        acc[RE(1, c)] += x1r;
        acc[IM(1, c)] += x1i;
        tot[c] += z0;
        tot[3 + c] += z1;
        // spins 2 and 3: chi1, chi0 (mu = 0, 1) or chi0, chi1 (mu = 2); with the factor i of mu = 0, 2 re and im change places
        const unsigned y0 = mu == 1 ? z0 : __byte_perm(z0, 0, 0x1032), y1 = mu == 1 ? z1 : __byte_perm(z1, 0, 0x1032);
        tot[6 + c] += mu == 2 ? y0 : y1;
        tot[9 + c] += mu == 2 ? y1 : y0;
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

// Resident blocks per SM: 4 (128 registers). Before the size test 3 (168 registers) was 2% faster at 32^3 x 64 (425
// against 435 us), but at 16^3 x 32 it leaves 56 of the 512 blocks to a second wave.
constexpr int HOP64_BLOCKS = 4;

// Bounds: 491 us at 32^3 x 64, where the same hop in FP64 arithmetic
// (hop_kernel<double, 18>) takes 1437, all of it FP64 pipe. A warp issues about
// 9600 instructions per 32 sites, 1728 of them wide integer multiply-adds: the
// multiplier pipe is busy 58% of the time and the schedulers 51%, at 15 warps
// per SM waiting on results and loads (profiles/hop64_clover_corr.md). The 1.7
// GB that it moves take 0.25 ms. The size test is 56 us of it, the exponent
// without a spare binade 10.
//
// The eight directions run as one loop body rather than unrolled: unrolled,
// the straight-line code ran at the rate of the instruction cache (770 us,
// against 435 without the size test, as the other figures here).
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

    // whole warps stay in the loop (hop64_sites); lanes beyond the last site do it once more and store nothing
    for (int i0 = sl.b * blockDim.x + threadIdx.x; i0 < sweep_end(Vh); i0 += sl.nb * blockDim.x) {
        const int h = min(i0, Vh - 1);
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
        unsigned tot[12];      // lower bounds of the sizes of each component's products, summed over the directions
#pragma unroll
        for (int i = 0; i < 12; ++i) tot[i] = 0;
        int E = 0;             // exponent of acc; 0 while every neighbour so far was zero
        bool bad = false;      // the site takes FP64 arithmetic
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
                if (E) {
                    const int sh = min(En - E, 63), shs = min(sh, 16);
                    const unsigned keep = (0xFFFFu >> shs) * 0x10001u;
#pragma unroll
                    for (int i = 0; i < 24; ++i) acc[i] >>= sh;
#pragma unroll
                    for (int i = 0; i < 12; ++i) tot[i] = (tot[i] >> shs) & keep;
                }
                E = En;
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
            int h0[12], h1[12], ht[12];   // ht: h in units of 2^30
            const bool rot = mu != 1;
            const int s = (d & 1) ? -1 : 0, s1 = mu == 0 ? s : ~s;
#pragma unroll
            for (int u = 0; u < 6; ++u) {
                const int mi = u < 3 ? s : s1, mr = rot ? ~mi : mi;
                const fx::Fixed pr = fx::fixed(p[u].y, p[u].x, E), pi = fx::fixed(p[u].w, p[u].z, E);
                const fx::Fixed qr = fx::fixed(rot ? q[u].w : q[u].y, rot ? q[u].z : q[u].x, E);
                const fx::Fixed qi = fx::fixed(rot ? q[u].y : q[u].w, rot ? q[u].x : q[u].z, E);
                const long long re = fx::sum(pr, fx::signed_by(qr, mr)), im = fx::sum(pi, fx::signed_by(qi, mi));
                fx::digits(re, h0[2 * u], h1[2 * u]);
                fx::digits(im, h0[2 * u + 1], h1[2 * u + 1]);
                ht[2 * u] = (int)(re >> 30);
                ht[2 * u + 1] = (int)(im >> 30);
            }
            // sizes of the half spinor, column by column: real parts, imaginary parts
            const unsigned zr0 = sizes(ht[0], ht[2], ht[4]), zi0 = sizes(ht[1], ht[3], ht[5]);
            const unsigned zr1 = sizes(ht[6], ht[8], ht[10]), zi1 = sizes(ht[7], ht[9], ht[11]);
            cp_async_wait<1>();
            long long x[12];   // U h: column k, row c, (re, im) at 6 k + 2 c
            unsigned z[6];     // sizes of its products
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
                const unsigned ur = sizes(l1[0], l1[2], l1[4]), ui = sizes(l1[1], l1[3], l1[5]);
                z[c] = __dp4a(ui, zi0, __dp4a(ur, zr0, 0u)) + (__dp4a(ui, zr0, __dp4a(ur, zi0, 0u)) << 16);
                z[3 + c] = __dp4a(ui, zi1, __dp4a(ur, zr1, 0u)) + (__dp4a(ui, zr1, __dp4a(ur, zi1, 0u)) << 16);
                fx::row_mul(l0, l1, n0, n1, h0, h1, x[2 * c], x[2 * c + 1]);
                fx::row_mul(l0, l1, n0, n1, h0 + 6, h1 + 6, x[6 + 2 * c], x[6 + 2 * c + 1]);
            }
            switch (d) {
            case 0: rebuild_fixed(0, true, x, z, acc, tot); break;
            case 1: rebuild_fixed(0, false, x, z, acc, tot); break;
            case 2: rebuild_fixed(1, true, x, z, acc, tot); break;
            case 3: rebuild_fixed(1, false, x, z, acc, tot); break;
            case 4: rebuild_fixed(2, true, x, z, acc, tot); break;
            case 5: rebuild_fixed(2, false, x, z, acc, tot); break;
            case 6: rebuild_fixed(3, true, x, z, acc, tot); break;
            default: rebuild_fixed(3, false, x, z, acc, tot); break;
            }
        }
        cp_async_wait<0>();      // a site left early may have a copy in flight
        if (E) {                 // the size test of every real (fixed64.cuh)
            unsigned least = tot[0];
#pragma unroll
            for (int i = 1; i < 12; ++i) least = __vminu2(least, tot[i]);
            bad = bad || (least & 0xFFFFu) < fx::SIZE_MIN || (least >> 16) < fx::SIZE_MIN;
        }
        double o[24];
#pragma unroll
        for (int i = 0; i < 24; ++i) o[i] = fx::to_double(acc[i], E);
        if (__any_sync(0xFFFFFFFFu, bad)) {
            double t[24];
            hop64_sites(P, vin, h, bad, t);
            if (bad)
                for (int i = 0; i < 24; ++i) o[i] = t[i];
        }
        if (i0 < Vh) hop_epilogue<double, EPI, RED, MAT>(P, vout, vy, vz, vrs, h, o, part, false);
    }
    if constexpr (RED != RED_NONE) grid_reduce<NS, RedStage<RED>::HINT>(part, P.rc, sl);
}

#undef RE
#undef IM

}  // namespace wd

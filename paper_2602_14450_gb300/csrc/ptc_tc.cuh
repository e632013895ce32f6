// First pass of the collapsed learned preconditioner on the 5th-generation
// tensor cores (tcgen05, kind::f16 with BF16 operands, FP32 accumulation in
// tensor memory).
//
// For every odd site y and colour a, the eight transports of the input,
// x[d1][t] = (T_{1+d1} psi)(y)_{t,a} (d1 = 0..7, spin t), are mixed into the
// eight intermediate fields phi_{1+d2}(y)_{s,a} = sum_{d1,t} V[1+d2][1+d1]_{st} x[d1][t].
// Written over the reals this is, per (site, colour) row, a 64-vector
// (d1, t, re/im) times a fixed 64 x 64 matrix -- a dense contraction of
// 3 * V/2 rows, K = 64, N = 64:
//   D[m][n] = sum_k A[m][k] B[n][k],  k = 8 d1 + 2 t + c,  n = 8 d2 + 2 s + c',
//   B = [[Re V, -Im V], [Im V, Re V]] in that index order.
// One CTA takes 128 odd sites: its 128 threads compute the transports (one site
// each, FP32 arithmetic) and write them, rounded to BF16, as three M = 128 x
// K = 64 operand tiles (one per colour); one thread issues the MMAs
// (M = 128, N = 64, 4 x K = 16 per colour); each warp reads its 32 rows back
// (tcgen05.ld) and stores phi colour-major: unit a of field d2 holds
// (s = 0..3, re/im) of colour a. Colours 0 and 1 are issued together into two
// 64-column accumulators and colour 2 follows into the first as soon as it has
// been read, so a tile waits for the tensor core once and synchronises three
// times. M with one accumulator, a wait and two barriers per colour, and with
// two (us, both passes): 16^3 x 32 38.6 / 38.8, 20^3 x 40 69.3 / 68.7,
// 24^3 x 48 121.3 / 120.0, 38 x 30 x 28 x 28 153.4 / 148.7, 32^3 x 64
// 317.6 / 317.1.
//
// Operand layout in shared memory: the no-swizzle K-major canonical form of
// 8-row x 16-byte core matrices. Element (m, k) of a tile with K = 64 sits at
// byte ((m / 8) * 8 + k / 8) * 128 + (m % 8) * 16 + (k % 8) * 2: the K-adjacent
// core-matrix stride (leading byte offset) is 128 and the M-adjacent one
// (stride byte offset) 1024; the K = 16 slice j starts 256 j bytes in.
//
// Every wait is bounded: on expiry the kernel raises *err, still waits (bounded)
// for its own MMAs, frees its tensor memory and returns.
#pragma once

#include <cstdint>

namespace wd {

namespace tc {

constexpr int TILE_M = 128;                  // sites per CTA tile
constexpr int K = 64, N = 64;                // real K and N of the contraction
constexpr int A_TILE_BYTES = TILE_M * K * 2; // one colour's operand tile (16 KB)
constexpr int B_BYTES = N * K * 2;           // 8 KB
constexpr int SMEM_BYTES = 3 * A_TILE_BYTES + B_BYTES + 64;
constexpr int TMEM_COLS = 128;              // two accumulators; three CTAs an SM take 384 of its 512 columns
constexpr unsigned WAIT_LIMIT = 1u << 22;    // try_wait rounds before giving up (the default)

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Byte offset of element (row, k) in a no-swizzle K-major tile with K = 64.
__host__ __device__ constexpr uint32_t kmajor_offset(int row, int k) {
    return (uint32_t)(((row >> 3) * 8 + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// Shared-memory matrix descriptor: start address, leading (K-adjacent) and
// stride (M/N-adjacent) core-matrix offsets, version 1, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
                           ((uint32_t)(TILE_M >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(IDESC), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void bar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// Wait for the phase with the given parity to complete; false when `limit`
// try_wait rounds ran out (limit 0: give up at once, without a round).
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity, unsigned limit = WAIT_LIMIT) {
    const uint32_t a = smem_addr(bar);
    for (unsigned i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 32 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

}  // namespace tc

// First pass (odd sites) of the collapsed M with the mixing on tensor cores.
// in_e: FP16 even-site input; phi: 8 BF16 odd-site fields (colour-major
// units), pvs units apart; links_o: FP16 12-real gathered links of the odd
// parity; V: collapsed spin weights [k2][k1][s][t]. Block size 128.
template <typename TIN, typename LT, int R>
__global__ void __launch_bounds__(128, 3) k_ptc_s1_tc(Geom g, const uint4* in_e, uint4* phi, long long pvs,
                                                      const uint4* links_o, const float2* V, const SolverState* guard,
                                                      int* err, unsigned wait_rounds) {
    // wait_rounds = the limit of the MMA waits + 1; 0 = the default limit
    const unsigned limit = wait_rounds ? wait_rounds - 1 : tc::WAIT_LIMIT;
    using namespace tc;
    if (guarded(guard, GUARD_INNER)) return;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* A = smem;                              // 3 colour tiles
    unsigned char* B = smem + 3 * A_TILE_BYTES;
    uint64_t* bar = reinterpret_cast<uint64_t*>(B + B_BYTES);   // one per accumulator
    uint32_t* tslot = reinterpret_cast<uint32_t*>(B + B_BYTES + 16);
    const int tid = threadIdx.x, warp = tid >> 5;

    // B[n][k] from V: n = 8 d2 + 2 s + c', k = 8 d1 + 2 t + c.
    for (int i = tid; i < N * K; i += blockDim.x) {
        const int n = i / K, k = i % K;
        const int d2 = n >> 3, s = (n >> 1) & 3, co = n & 1;
        const int d1 = k >> 3, t = (k >> 1) & 3, ci = k & 1;
        const float2 v = V[((1 + d2) * 9 + 1 + d1) * 16 + 4 * s + t];
        const float val = co == 0 ? (ci == 0 ? v.x : -v.y) : (ci == 0 ? v.y : v.x);
        *reinterpret_cast<__nv_bfloat16*>(B + kmajor_offset(n, k)) = __float2bfloat16_rn(val);
    }
    if (tid == 0) {
        bar_init(bar, 1);
        bar_init(bar + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(tslot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    fence_proxy_async();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t lane_base = (uint32_t)(32 * warp) << 16;
    const uint32_t a_base = smem_addr(A), b_base = smem_addr(B);
    uint32_t issued[2] = {0, 0};   // commits on each barrier so far; the last one completes the phase of parity (n - 1) & 1
    bool failed = false;
    auto issue = [&](int a) {      // colour a into accumulator a & 1
        if (tid == 0) {
#pragma unroll
            for (int j = 0; j < K / 16; ++j) {
                const uint64_t ad = smem_desc(a_base + a * A_TILE_BYTES + 256 * j, 128, 1024);
                const uint64_t bd = smem_desc(b_base + 256 * j, 128, 1024);
                tc::mma_bf16(tmem + 64 * (a & 1), ad, bd, j > 0 ? 1u : 0u);
            }
            mma_commit(bar + (a & 1));
        }
        ++issued[a & 1];
    };
    // waits for an accumulator's last MMA and reads this thread's row of it; false when the wait ran out in this warp
    auto read = [&](int acc, float (&v)[64]) {
        const bool landed = __all_sync(0xffffffffu, bar_wait(bar + acc, (issued[acc] - 1) & 1, limit));
        if (landed) {
            fence_after();
            tmem_ld32(tmem + lane_base + 64 * acc, v);
            tmem_ld32(tmem + lane_base + 64 * acc + 32, v + 32);
            tmem_ld_wait();
        }
        return landed;
    };

    const int ntiles = (g.Vh + TILE_M - 1) / TILE_M;
    for (int tile = blockIdx.x; tile < ntiles && !failed; tile += gridDim.x) {
        const int h = tile * TILE_M + tid;
        const bool ok = h < g.Vh;
        static_assert(R == 12 && sizeof(TIN) == 2 && sizeof(LT) == 2, "FP16 input, FP16 12-real links");
        // transports -> BF16 operand rows (zero rows past the end); each
        // direction's neighbour and link units are loaded one direction ahead
        int nbr[8];
        unsigned wm = 0;
        uint4 fu[2][3], lu[2][2];
        if (ok) {
            wm = site_neighbours(g, 1, h, nbr);
#pragma unroll
            for (int u = 0; u < 3; ++u) fu[0][u] = __ldg(in_e + (size_t)u * g.Vh + nbr[0]);
            load_link_units<LT>(links_o, g.Vh, h, 0, lu[0]);
        }
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            float t[24];
            if (ok) {
                if (d + 1 < 8) {
#pragma unroll
                    for (int u = 0; u < 3; ++u) fu[(d + 1) & 1][u] = __ldg(in_e + (size_t)u * g.Vh + nbr[d + 1]);
                    load_link_units<LT>(links_o, g.Vh, h, d + 1, lu[(d + 1) & 1]);
                }
                float f[24], m[18];
#pragma unroll
                for (int u = 0; u < 3; ++u)
#pragma unroll
                    for (int i = 0; i < 8; ++i) f[8 * u + i] = Unit<TIN>::get(fu[d & 1][u], i);
                link_from_units<LT>(lu[d & 1], d, m);
                colour_mul(m, f, t);
                if (((wm >> d) & 1u) && g.bc[d >> 1] < 0) {
#pragma unroll
                    for (int i = 0; i < 24; ++i) t[i] = -t[i];
                }
            } else {
#pragma unroll
                for (int i = 0; i < 24; ++i) t[i] = 0.f;
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {   // k = 8 d + 2 s + c: spins 0..3 of colour a, (re, im)
                uint4 w;
                w.x = pack_bf16(t[2 * (0 + a)], t[2 * (0 + a) + 1]);
                w.y = pack_bf16(t[2 * (3 + a)], t[2 * (3 + a) + 1]);
                w.z = pack_bf16(t[2 * (6 + a)], t[2 * (6 + a) + 1]);
                w.w = pack_bf16(t[2 * (9 + a)], t[2 * (9 + a) + 1]);
                *reinterpret_cast<uint4*>(A + a * A_TILE_BYTES + kmajor_offset(tid, 8 * d)) = w;
            }
        }
        fence_proxy_async();
        fence_before();
        __syncthreads();
        fence_after();

        auto store = [&](int a, const float (&v)[64]) {   // rows past the end are not stored
            if (!ok) return;
#pragma unroll
            for (int d2 = 0; d2 < 8; ++d2) {
                uint4 w;
                w.x = pack_bf16(v[8 * d2], v[8 * d2 + 1]);
                w.y = pack_bf16(v[8 * d2 + 2], v[8 * d2 + 3]);
                w.z = pack_bf16(v[8 * d2 + 4], v[8 * d2 + 5]);
                w.w = pack_bf16(v[8 * d2 + 6], v[8 * d2 + 7]);
                phi[(size_t)d2 * pvs + (size_t)a * g.Vh + h] = w;
            }
        };
        issue(0);
        issue(1);
        float row[64];
        bool landed = read(0, row);
        fence_before();
        failed = __syncthreads_or(!landed);      // uniform across the CTA: accumulator 0 has been read
        fence_after();
        if (!failed) {
            issue(2);
            store(0, row);
            landed = read(1, row);
            if (landed) store(1, row);
            const bool last = read(0, row);
            if (last) store(2, row);
            fence_before();
            failed = __syncthreads_or(!landed || !last);   // all read, and the operand tiles are free again
            fence_after();
        }
        if (failed && tid == 0 && err) *(volatile int*)err = 1;
    }
    if (failed && tid == 0) {   // default bound: let MMAs still in flight finish
        for (int i = 0; i < 2; ++i) bar_wait(bar + i, (issued[i] - 1) & 1);
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

}  // namespace wd

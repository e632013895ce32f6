// Host-side launchers of the device kernels, one instantiation per storage
// type (translation units ops_f64.cu, ops_f32.cu, ops_f16.cu, ops_bf16.cu).
//
// Every vector argument may hold a batch of `nrhs` right-hand sides stored
// back to back: right-hand side r of a packed parity vector starts `vs`
// 16-byte units after right-hand side r - 1 (vs = units per site * V/2 for a
// tightly packed batch). Scalar state, reduction partials and tickets are
// arrays over right-hand sides (see RedCtx).
#pragma once

#include "common.cuh"

namespace wd {

// s += a b + c d and s += a b - c d. FP64 takes two fused multiply-adds: its pipe (2 per cycle and SM) bounds the
// FP64 vector kernels and reductions, and the expression as written is three operations there.
template <typename C> __device__ __forceinline__ void add_products(C& s, C a, C b, C c, C d) { s += a * b + c * d; }
template <> __device__ __forceinline__ void add_products<double>(double& s, double a, double b, double c, double d) {
    s = fma(c, d, fma(a, b, s));
}
template <typename C> __device__ __forceinline__ void sub_products(C& s, C a, C b, C c, C d) { s += a * b - c * d; }
template <> __device__ __forceinline__ void sub_products<double>(double& s, double a, double b, double c, double d) {
    s = fma(-c, d, fma(a, b, s));
}
// The same as two fused multiply-adds in FP32 (the dot products of the FP16-arithmetic hop): two roundings instead of
// three and two operations instead of three. One inner iteration of the FP16-mixed solve at 32^3 x 64: 931.1 us with
// the expressions above, 926.6 us so; at 24^3 x 48 376.4 and 375.6 us (three runs each, within 1.3 us).
__device__ __forceinline__ void add_fused(float& s, float a, float b, float c, float d) { s = fma(c, d, fma(a, b, s)); }
__device__ __forceinline__ void sub_fused(float& s, float a, float b, float c, float d) { s = fma(-c, d, fma(a, b, s)); }

enum Epi { EPI_H = 0, EPI_Y = 1, EPI_YZ = 2 };
enum Red { RED_NONE = 0, RED_RSV = 1, RED_TS = 2, RED_NORM = 3 };
// Rescaling of r in the x/r-update kernel k_xr (Alg. 4): none, norms for a separate k_scale pass, or fused.
enum XrMode { XR_PLAIN = 0, XR_NORMS = 1, XR_FUSED = 2 };

struct HopParams {
    Geom g;
    int parity;             // parity of the output sites
    int nrhs;               // right-hand sides in the batch (>= 1)
    long long vs;           // units between right-hand sides of every spinor argument
    const uint4* links;     // gathered links of the output parity (shared by all rhs)
    const uint4* in;        // input spinor on parity 1 - parity
    uint4* out;             // output spinor on `parity`
    const uint4* y;         // epilogue operands on `parity`
    const uint4* z;
    const uint4* rstar;     // RED_RSV: sum conj(rstar) out
    double a, b, c;         // out = a * H in + b * y + c * z
    RedCtx rc;              // reduction target (partials, ticket, state, stage)
    const SolverState* guard;  // per-rhs state consulted by the guard
    int guard_kind;            // GuardKind
    int* err;                  // set to 1 by a kernel whose bounded wait gave up (may be null)
    const uint4* mat;          // site-local 12 x 12 complex block of the output parity (chiral packing,
                               // storage T) applied to the hop: out = M (a H in) + b y + c z; null = none
    int variant[2];            // kernel variant (hop_variant() numbering) without / with a fused
                               // reduction; 0 = the process default
    int block[2];              // threads per block, likewise; 0 = the process default
    int arith16;               // FP16 storage only: 1 = the hopping sum in FP16 arithmetic (hop16_kernel)
    int acc_exp;               // hop16_kernel: exponent of its accumulator scale (set by the launcher)
    unsigned wait_rounds;      // limit of a bounded device wait + 1 (wd_set_wait_limit); 0 = the default limit
    int rhs_group[2];          // FP16 arithmetic: right-hand sides per thread (hop16m_kernel) without / with a
                               // fused reduction; 0 or 1 = one (hop16_kernel); must divide nrhs to be used
    int rhs_smem[2];           // ... and 1 = the site's links in shared memory instead of registers
    int rev;                   // 1 = take the sites from the last to the first (sweep_site; FP16 arithmetic)
    int fixed64;               // FP64, 18-real: the links are fixed-point digits (hop64_kernel)
    const double* U64;         // ... and the FP64 links in the host layout, for sites that take FP64 arithmetic
    int spt;                   // FP16 arithmetic, plain hop: sites per thread (grid-stride; 0 or 1 = one site)
};

// Largest number of blocks a reducing kernel uses per right-hand side.
constexpr int MAX_RED_BLOCKS = 8192;
constexpr int MAX_RED_SUMS = 4;
static_assert(MAX_RED_BLOCKS * MAX_RED_SUMS == RED_STRIDE, "partials layout");

// Units of 16 bytes per site of the gathered links of one parity.
int link_units(int prec, int recon);
// Units of 16 bytes per site of a spinor.
int spinor_units(int prec);

// Vector kernels: n = sites per parity, vs = units between right-hand sides
// (vs64 for FP64 vectors), st = state array, g = guard kind.
template <typename T> struct Ops {
    static cudaError_t hop(int recon, int epi, int red, const HopParams& P, cudaStream_t s);
    // variant and threads per block of a hop whose HopParams choose none (environment, else by rule)
    static void default_hop(int recon, const Geom& g, bool reducing, int* variant, int* block);
    // rev: order of the sites (sweep_site)
    static cudaError_t pupdate(int n, int nrhs, long long vs, uint4* p, const uint4* v, const uint4* r,
                               const SolverState* st, int rev, cudaStream_t s);
    static cudaError_t supdate(int n, int nrhs, long long vs, uint4* r, const uint4* v, const SolverState* st,
                               int rev, cudaStream_t s);
    // mode: XrMode
    static cudaError_t xr(int mode, int n, int nrhs, long long vs, uint4* x, uint4* r, const uint4* p,
                          const uint4* t, const uint4* rstar, const uint4* xr_src, const uint4* xp_src,
                          SolverState* st, RedCtx rc, int rev, cudaStream_t s);
    static cudaError_t scale(int n, int nrhs, long long vs, uint4* r, uint4* x, const uint4* rstar, SolverState* st,
                             RedCtx rc, cudaStream_t s);
    static cudaError_t rescale_in(int n, int nrhs, long long vs, long long vs64, const uint4* r64, uint4* r,
                                  uint4* rstar, int ftz, SolverState* st, RedCtx rc, cudaStream_t s);
    static cudaError_t correct(int n, int nrhs, long long vs, long long vs64, uint4* x64, const uint4* xt,
                               const SolverState* st, cudaStream_t s);
    static cudaError_t norm2(int n, int nrhs, long long vs, const uint4* v, RedCtx rc, int guard_kind,
                             cudaStream_t s);
    // xo = eta + kappa t and the sum of |eta - xo + kappa t|^2 (Eq. 5 with t = H_oe xi_e)
    static cudaError_t odd_reconstruct(int n, int nrhs, long long vs, double kappa, const uint4* eta, const uint4* t,
                                       uint4* xo, RedCtx rc, cudaStream_t s);
    // out = M in, or with `one` in + M in, with M in the chiral packing (80 reals per site, see mat_mul_chiral)
    static cudaError_t apply_chiral(int n, int nrhs, long long vs, const uint4* mat, const uint4* in, uint4* out,
                                    bool one, cudaStream_t s);
    // chiral packing in storage T from FP64
    static cudaError_t chiral_from64(int n, const uint4* src64, uint4* dst, cudaStream_t s);
    static cudaError_t pack(const Geom& g, int parity, const double* lex, uint4* out, cudaStream_t s);
    static cudaError_t unpack(const Geom& g, int parity, const uint4* in, double* lex, cudaStream_t s);
    // fixed64: FP64 18-real links as fixed-point digits (SU(3) links only; fixed64.cuh)
    static cudaError_t build_links(int recon, const Geom& g, int parity, const double* U, uint4* out, bool fixed64,
                                   cudaStream_t s);
};

cudaError_t launch_unitarity(int nlinks, const double* U, unsigned long long* out, cudaStream_t s);

int num_sms();
inline int stream_blocks(int n, int block) {
    long g = ((long)n + block - 1) / block;
    return g < 1 ? 1 : (int)g;
}

// Threads per block of a launch over n items for each of nrhs right-hand sides: `block`, or on a small lattice a
// half, quarter, ... of it down to one warp until every SM has a block. A kernel of 16 blocks of 128 threads (8^4)
// otherwise runs on 16 of the 152 SMs.
inline int spread_block(int n, int nrhs, int block) {
    while (block > 32 && (long)stream_blocks(n, block) * nrhs < num_sms()) block /= 2;
    return block;
}

constexpr int HOP64_THREADS = 128;   // largest block of the fixed-point FP64 hop

// Block size of every vector kernel. The hop kernels take theirs from
// HopParams::block (set by wd_tune), else from the environment (WD_HOP_BLOCK =
// 64 or 128), else by rule (default_block).
constexpr int VEC_BLOCK = 256;
int hop_block();     // the environment's, 0 = none
// Hop kernel variant, from HopParams::variant, else from the environment
// (WD_HOP_KERNEL), else by rule (default_variant):
// 4 = one site per thread, neighbour and link loads issued one direction
// ahead; 1 = one site per thread without the look-ahead; 6 = as 4 with the
// SU(3) products on FP32x2 pairs; for FP32-arithmetic storage 2 = two sites per
// thread with packed FP32x2 math; for 16-bit storage 3 = tiles staged in shared
// memory by bulk copies and, with 12-real links, 5 = persistent threads
// streaming their operands through a per-thread two-slot ring of asynchronous
// copies in shared memory.
int hop_variant();   // the environment's, 0 = none
// Directions ahead that the FP16-arithmetic hop loads its neighbour spinors
// (environment WD_HOP16_AHEAD = 1 or 2, default 2: 3% faster at 32^3 x 64).
int hop16_ahead();

}  // namespace wd

// gs_common.cuh -- internal definitions shared by the CUDA translation units of libgsmri.
// Not part of the public ABI (include/gs_api.h is).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gs_api.h"

namespace gs {

// ------------------------------------------------------------------ render record
// Per-Gaussian record (20 floats = 5 float4, 80 bytes) written by the preprocess kernel and
// staged into shared memory by the render kernels. Coordinates are voxel-index space: voxel
// (i, j, k) sits at (i, j, k). The mean mu' = (mu - o) / h - 1/2 is a float head plus a
// float tail (double-float arithmetic), stored negated, so d = (i + (-head)) + (-tail) =
// (i - head) - tail is accurate to one rounding of d even at large coordinates, and the
// (y, z) components of a row's offset are one packed pair of additions.
// The exponent q = (log2 e / 2) d^T Sigma'^{-1} d (Sigma' the covariance in voxel units, the
// Gaussian kernel is 2^-q) is stored by completing the square along x:
//     q(dx, dy, dz) = S(dy, dz) + (sa (dx - dx*(dy, dz)))^2,
//     S(dy, dz) = Pyy dy^2 + P2yz dy dz + Pzz dz^2   (the minimum of q along the x-row),
//     dx*(dy, dz) = c1 dy + c2 dz                      (where that minimum is reached);
// (P2yz, c2) and (Pyy, c1) sit side by side, so (Pyy dy + P2yz dz, c1 dy + c2 dz) is one
// packed multiply and one packed FMA.
// With M = sqrt(log2 e / 2) diag(1/s) R^T H (columns m0, m1, m2, the whitened steps of one
// voxel along x, y, z): sa = |m0| (the whitened length of one voxel step along x),
// c_j = -(m_j . m0) / |m0|^2, and S is the Gram form of m1, m2 with their components along m0
// removed. Every term of this form has the size of q itself
// for voxels inside the ellipsoid, so FP32 keeps its accuracy for strongly anisotropic
// Gaussians, and the value at a voxel depends only on the voxel and the Gaussian.
// rho4 bounds |M (p - c)| over a 4 x 4 x 4 voxel footprint around its centre c:
// |M d|^2 <= sum_jk |m_j . m_k| |d_j| |d_k| <= (3/2)^2 sum_jk |m_j . m_k| (culling).
// ext_k = 1.01 trunc_sigma sigma_k + 3/2 + 10^-3 (sigma_k the standard deviation along axis k
// in voxels) bounds the offset of a 4^3 footprint's centre from the mean when the truncated
// ellipsoid reaches one of its voxels (culling).
enum RecField : int {
    R_NMHX = 0, R_NMLX = 1,                 // -(mu' head, tail) along x
    R_NMHY = 2, R_NMHZ = 3,                 // -mu' head along y, z
    R_NMLY = 4, R_NMLZ = 5,                 // -mu' tail along y, z
    R_P2YZ = 6, R_C2 = 7,                   // dz coefficients of the row terms (S, dx*)
    R_PYY = 8, R_C1 = 9,                    // their dy coefficients
    R_PZZ = 10, R_SA = 11,                  // dz^2 coefficient of S; sa = |m0|
    R_EXTX = 12,                            // box half-extent along x (see below)
    R_RHO4 = 13,                            // footprint radius (see above)
    R_EXTY = 14, R_EXTZ = 15,               // box half-extents along y, z
    R_VR = 16,                              // v * r
    R_R = 17,                               // r
    R_V = 18,                               // v
    REC_FLOATS = 20
};
constexpr int REC_F4 = REC_FLOATS / 4;

// Render-space gradient accumulated per Gaussian by the adjoint kernel (12 floats):
// m1 = sum G d (3), m2 = sum G d d^T (xx, yy, zz, xy, xz, yz), dv, dr, pad, where
// G = dL/dw * w for every contributing pair (see gs_render.cu).
enum GradField : int {
    G_M1X = 0, G_M1Y = 1, G_M1Z = 2,
    G_M2XX = 3, G_M2YY = 4, G_M2ZZ = 5, G_M2XY = 6, G_M2XZ = 7, G_M2YZ = 8,
    G_DV = 9, G_DR = 10, G_PAD = 11,
    GRAD_FLOATS = 12
};

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kHalfLog2e = 0.7213475204444817f;  // (1/2) log2(e)

// Brick-range brange layout [N, 8].
enum BrangeField : int { B_LOX = 0, B_LOY, B_LOZ, B_HIX, B_HIY, B_HIZ, B_CNT, B_VALID };

// Streaming multiprocessors of the GPU that the grids and the sizes of the dispatch rules are made for.
constexpr int kSms = 152;

// ------------------------------------------------------------------ sort constants
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;  // 2048 keys per tile
// First-pass tiles of more than kSortTile pairs take rounds of 2,304: a round costs 7 us or more whether
// full or nearly empty, and tiles of 256 Gaussians with 8.2-8.5 pairs each needed a second one (833,333
// Gaussians, 6.83M pairs, whole binning 182 -> 171 us; 100,000 with 7.1 pairs 36.7 -> 35.5; 4M with 26
// 2.40 -> 2.36 ms). Used for all tiles, 0.2 % of a step at 5.6-6.5 pairs, which fill one round either
// way. 10 and more items spill at 64 registers; with the keys read again from shared memory instead, 10
// (12) take 171 (171) us and 2.34 (2.28) ms, but 69.3 (69.4) us against 67.5 at 375,000 with 5.6 pairs
// and 89.9 (89.3) against 88.8 at 500,000.
constexpr int kFirstItems = 9;
// A tile's own block places at most first_part(P) of its pairs; what is left of a heavier tile is taken
// in parts of that size by further blocks, each of which first counts the digits of the tile's pairs
// before its part (by rows of the boxes). So a block's serial work follows the pairs in all, not the
// widest Gaussians: four rounds at least, and no less than twice an even share of the pairs among the
// resident blocks, so that clouds whose tiles are all alike are not cut up (with one share 12.3M pairs in
// 391 tiles 490 -> 525 us).
constexpr int kFirstRound = kSortThreads * kFirstItems;
constexpr int kFirstMinPart = 4 * kFirstRound;
constexpr int kScatterWave = kSms * 4;  // resident scatter blocks
constexpr int kFirstParts = kScatterWave / 2;
__host__ __device__ inline int64_t first_part(int64_t pairs) {
    const int64_t share = (pairs / kFirstParts / kFirstRound + 1) * kFirstRound;  // > pairs / kFirstParts
    return share > kFirstMinPart ? share : kFirstMinPart;
}
constexpr int kMaxRadixBits = 9;
constexpr int kMaxDigits = 1 << kMaxRadixBits;
// Gaussians per block of the preprocess and emission kernels. A cloud that would fill no more than one
// block of 256 per SM is spread over more SMs in tiles of 64: 6,000 clustered Gaussians, 119,000 pairs,
// one radix pass 18.2 -> 7.8 us, preprocess 6.9 -> 6.3; 30,000 lattice Gaussians 8.1 -> 6.5 us; the
// largest such cloud gains least.
constexpr int64_t kSmallCloud = kSms * 256;
inline int gauss_tile(int64_t n_gauss) { return n_gauss <= kSmallCloud ? 64 : 256; }

constexpr int kL1Blocks = 1024;  // fixed block count of the L1 reduction (deterministic)

constexpr int64_t kMaxCapacity = (int64_t(1) << 31) - 4096;

// ------------------------------------------------------------------ workspace layout
struct Workspace {
    int32_t* keys[2];        // brick keys between the radix passes; the second of each pair is
    int2* vals[2];           // bound for three passes and more. vals: (Gaussian-major position, id)
    int32_t* hist0;          // first pass's digit counts: one row per digit, a column per
                             // Gaussian tile (row stride stride0)
    int32_t* hist[2];        // later passes': a column per kSortTile pairs (row stride stride1)
    int32_t* rowtot;         // [kMaxDigits] totals of the digits of the pass being scanned
    long long* blk_base;     // [Gaussian tiles + 2] pairs of each tile, then their exclusive sums (one more
                             // entry than tiles) and the heaviest tile's pairs
    int64_t stride0, stride1;
    int32_t key_bits, radix_passes;
    float* part;             // [capacity, 12] per-pair partial gradients (deterministic mode)
    float* gacc;             // [n_gauss, 12] render-space gradient per Gaussian
    float2* aip;             // [n_voxels] (alpha, alpha I'), alpha = dL/dI / max(W, eps)
    float* l1_part;          // [kL1Blocks]
    int32_t* ticket;         // finished blocks of the fitting step's loss kernel, cleared by the
                             // binning's first scan
    size_t bytes;
};

// Stable LSD radix sort of the brick keys: as few passes of at most kMaxRadixBits bits as the
// keys need, with digit widths as equal as can be (16,384 bricks: 7 + 7 bits; 20,480: 7 + 8; 131,072: 9 + 8).
// Narrow digits give longer runs per tile and digit, and fewer count rows to scan. Unequal widths:
// the narrow ones first, whose pass has the more and the less full tiles (20,480 bricks, 4.72M pairs:
// 130 us against 134), but a 9-bit digit before an 8-bit one: lists over so many bricks are larger than
// L2, and the last pass, which stores three arrays of 4 bytes, then writes runs of eight pairs, whole
// sectors (131,072 bricks, 104M pairs: 2.39 ms against 2.48).
inline void radix_plan(int32_t n_bricks, int32_t* passes, int32_t* key_bits) {
    int need = 1;
    while ((int64_t(1) << need) < n_bricks) ++need;
    *passes = (need + kMaxRadixBits - 1) / kMaxRadixBits;
    *key_bits = need;
}

// Width of the digit of one of the passes.
inline int pass_bits(int key_bits, int passes, int pass) {
    const int narrow = key_bits / passes, wide = key_bits % passes;  // so many passes of narrow + 1 bits
    const bool is_wide = narrow + 1 == kMaxRadixBits ? pass < wide : pass >= passes - wide;
    return narrow + (is_wide ? 1 : 0);
}

// Who counts a later pass's digits: from this many Gaussians on a kernel of its own, over the output of
// the pass before; below, the scatter before itself, with an atomic per group of equal (tile, digit) in a
// warp.
// The launch costs 2 us; the atomics nothing where neighbours in the list are neighbours in space
// (lattice clouds, whose groups are large: 131,072 Gaussians, 0.71M pairs 36.4 us with them, 39.1
// without; 500,000: 88.6, 89.0; 1M: 130.4, 130.5) and 4 us per million pairs where they are not (1M
// random Gaussians, 6.83M pairs 184.3 us with them, 182.1 without; 4M clustered ones, 104M pairs 2.81 ms
// and 2.40 ms).
constexpr int64_t kCountCloud = 400000;

inline bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Carve (or size, if base == nullptr) the workspace. Returns false on overflow.
inline bool carve_workspace(void* base, int64_t n_gauss, int64_t capacity, int32_t n_bricks,
                            int64_t n_voxels, bool deterministic, Workspace* ws) {
    size_t off = 0;
    auto take = [&](size_t bytes) -> char* {
        size_t o = off;
        off = align_up(off + bytes, 256);
        return base ? static_cast<char*>(base) + o : nullptr;
    };
    const int64_t cap = capacity > 0 ? capacity : 1;
    const int64_t n = n_gauss > 0 ? n_gauss : 1;
    radix_plan(n_bricks, &ws->radix_passes, &ws->key_bits);
    // Counts and tiles are sized for the largest table of any smaller problem (fewer Gaussians in smaller
    // tiles; fewer bricks in fewer, wider digits), so that a workspace serves every smaller problem too.
    const int64_t nd0 = int64_t(1) << (ws->key_bits < kMaxRadixBits ? ws->key_bits : kMaxRadixBits);
    const int64_t nd1 = ws->radix_passes > 2 ? kMaxDigits : int64_t(1) << (ws->key_bits + 1) / 2;
    const int64_t small_tiles = ((n < kSmallCloud ? n : kSmallCloud) + 63) / 64, large_tiles = (n + 255) / 256;
    const int64_t max_tiles = small_tiles > large_tiles ? small_tiles : large_tiles;
    const int64_t g_tiles = (n + gauss_tile(n) - 1) / gauss_tile(n);
    ws->stride0 = (g_tiles + 3) / 4 * 4;  // rows are scanned in 16-byte pieces
    ws->stride1 = ((cap + kSortTile - 1) / kSortTile + 3) / 4 * 4;
    for (int k = 0; k < 2; ++k) {
        const bool used = k == 0 ? ws->radix_passes > 1 : ws->radix_passes > 2;
        ws->keys[k] = reinterpret_cast<int32_t*>(take(used ? sizeof(int32_t) * cap : 256));
        ws->vals[k] = reinterpret_cast<int2*>(take(used ? sizeof(int2) * cap : 256));
        ws->hist[k] = reinterpret_cast<int32_t*>(take(used ? sizeof(int32_t) * nd1 * ws->stride1 : 256));
    }
    ws->hist0 = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * nd0 * ((max_tiles + 3) / 4 * 4)));
    ws->rowtot = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * kMaxDigits));
    ws->blk_base = reinterpret_cast<long long*>(take(sizeof(long long) * (max_tiles + 2)));
    ws->part = reinterpret_cast<float*>(
        take(deterministic ? sizeof(float) * GRAD_FLOATS * cap : 256));
    ws->gacc = reinterpret_cast<float*>(take(sizeof(float) * GRAD_FLOATS * n));
    ws->aip = reinterpret_cast<float2*>(take(sizeof(float2) * (n_voxels > 0 ? n_voxels : 1)));
    ws->l1_part = reinterpret_cast<float*>(take(sizeof(float) * kL1Blocks));
    ws->ticket = reinterpret_cast<int32_t*>(take(sizeof(int32_t)));
    ws->bytes = off;
    return true;
}

// Division by an invariant positive integer d (T. Granlund and P. L. Montgomery, "Division by
// invariant integers using multiplication", PLDI 1994, the unsigned case): with
// l = ceil(log2 d) and m = floor(2^32 (2^l - d) / d) + 1, every 32-bit unsigned n has
// n / d = (t + ((n - t) >> s1)) >> s2, t = mulhi(m, n), s1 = min(l, 1), s2 = max(l - 1, 0):
// one high multiply, a subtraction and three shifts in place of a division sequence.
struct FastDiv {
    unsigned m;
    int s1, s2;
};

inline FastDiv make_fastdiv(unsigned d) {
    int l = 0;
    while ((1ull << l) < d) ++l;
    FastDiv f;
    f.m = static_cast<unsigned>(((1ull << 32) * ((1ull << l) - d)) / d + 1ull);
    f.s1 = l < 1 ? l : 1;
    f.s2 = l - 1 > 0 ? l - 1 : 0;
    return f;
}

// ------------------------------------------------------------------ helpers
struct BrickGeom {
    int nbx, nby, nbz;
    int bx, by, bz;
};

inline BrickGeom brick_geom(const gs_grid* g, const gs_config* c) {
    BrickGeom b;
    b.bx = c->brick[0];
    b.by = c->brick[1];
    b.bz = c->brick[2];
    b.nbx = (g->nx + b.bx - 1) / b.bx;
    b.nby = (g->ny + b.by - 1) / b.by;
    b.nbz = (g->nz + b.bz - 1) / b.bz;
    return b;
}

// Validation shared by the entry points. Returns GS_OK or GS_ERR_INVALID_ARG.
gs_status validate_grid_cfg(const gs_grid* g, const gs_config* c);

// Launch counter (every kernel launch site is followed by last_launch_status()).
void note_launch();

// ------------------------------------------------------------------ launch chaining
// Programmatic dependent launch (sm_90 and later): every kernel is launched with programmatic
// stream serialisation, so its launch overlaps the end of its predecessor on the stream, and
// its first statement (pdl_enter) waits until the predecessor has completed and its memory is
// visible; nothing is read or written before the wait. Kernels do not trigger their
// successors early (the trigger is implicit as their blocks exit): an early trigger measured
// slower in graph replays of the fitting step.
template <typename... P, typename... A>
inline void launch_k(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     A&&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    (void)cudaLaunchKernelEx(&c, k, static_cast<A&&>(args)...);  // errors: cudaGetLastError
}

// Launch error check -> gs_status; counts the launch it follows.
inline gs_status last_launch_status() {
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

gs_status resample_fwd_impl(const float* src, int32_t snz, int32_t sny, int32_t snx, float* dst,
                            int32_t dnz, int32_t dny, int32_t dnx, cudaStream_t st);
gs_status resample_adj_prep_impl(const float* dlr, int32_t lnz, int32_t lny, int32_t lnx,
                                 const float* I, const float* W, int32_t nz, int32_t ny, int32_t nx,
                                 float eps, float2* aip, cudaStream_t st);
// Fitting-step tails (gs_param.cu): chain without Adam; Adam with an optional device skip flag.
gs_status launch_chain_grad(const float* params, float* grad, const float* part,
                            const float* gacc, const gs_bins* bins, int64_t n,
                            const gs_grid* grid, const gs_config* cfg, cudaStream_t st);
gs_status launch_adam(float* params, const float* grad, float* m, float* v, int64_t n_gauss,
                      const gs_adam* hp, int32_t* d_step, const int32_t* d_skip,
                      cudaStream_t st);

}  // namespace gs

// ------------------------------------------------------------------ device math
#ifdef __CUDACC__
namespace gs {

// FP32 exponential of the binning specification: Cody-Waite argument reduction with a
// 15-bit head of ln 2 and a degree-7 Taylor polynomial in Horner form (W. J. Cody and
// W. Waite, "Software Manual for the Elementary Functions", 1980). Every operation is one
// explicitly rounded IEEE operation in a fixed order (no contraction), so the result is the
// same on any IEEE-754 implementation that follows the same sequence. |x| <= 30.
__device__ __forceinline__ float exp_cw(float x) {
    const float L2E = 1.44269502f;
    const float LN2_HI = 0.693145751953125f;
    const float LN2_LO = 1.42860677e-6f;
    float kf = floorf(__fadd_rn(__fmul_rn(x, L2E), 0.5f));
    float r = __fsub_rn(__fsub_rn(x, __fmul_rn(kf, LN2_HI)), __fmul_rn(kf, LN2_LO));
    float p = 1.0f / 5040.0f;
    p = __fadd_rn(__fmul_rn(p, r), 1.0f / 720.0f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f / 120.0f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f / 24.0f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f / 6.0f);
    p = __fadd_rn(__fmul_rn(p, r), 0.5f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f);
    p = __fadd_rn(__fmul_rn(p, r), 1.0f);
    int k = static_cast<int>(kf);
    float two_k = __int_as_float((k + 127) << 23);
    return __fmul_rn(p, two_k);
}

// First statement of every kernel: wait for the preceding kernel on the stream (see
// launch_k; a no-op for a launch without a programmatic dependency).
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// 2^x on the special-function unit (ex2.approx, flush-to-zero).
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Approximate square root (sqrt.approx, flush-to-zero); for bounds that carry a margin.
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Approximate reciprocal square root (rsqrt.approx, flush-to-zero); for bounds that carry a margin.
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Four values, as one 16-byte access (kVec) or one by one.
template <bool kVec>
__device__ __forceinline__ void load4(const float* src, float (&d)[4]) {
    if (kVec) {
        const float4 a = *reinterpret_cast<const float4*>(src);
        d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = src[k];
    }
}

template <bool kVec>
__device__ __forceinline__ void store4(float* dst, const float (&d)[4]) {
    if (kVec) {
        *reinterpret_cast<float4*>(dst) = make_float4(d[0], d[1], d[2], d[3]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) dst[k] = d[k];
    }
}

// Adjoint render's factors of one voxel (see k_bwd_prep).
__device__ __forceinline__ float2 adj_factor(float gI, float w, float iv, float eps) {
    const float al = gI / (w > eps ? w : eps);
    return make_float2(al, (w > eps) ? al * iv : 0.0f);
}

// dL/dI of kV (4 or 1) consecutive voxels from v on: as it is, or (kPrep) as the adjoint render's factors.
template <bool kPrep, int kV>
__device__ __forceinline__ void emit_voxels(int64_t v, const float (&acc)[kV], const float* __restrict__ Iv,
                                            const float* __restrict__ Wv, float eps, float* __restrict__ dsrc,
                                            float2* __restrict__ aip) {
    if constexpr (kPrep) {
        float w[kV], iv[kV];
        float2 a[kV];
        if constexpr (kV == 4) {
            load4<true>(Wv + v, w);
            load4<true>(Iv + v, iv);
        } else {
            w[0] = Wv[v];
            iv[0] = Iv[v];
        }
#pragma unroll
        for (int e = 0; e < kV; ++e) a[e] = adj_factor(acc[e], w[e], iv[e], eps);
        if constexpr (kV == 4) {
            reinterpret_cast<float4*>(aip + v)[0] = make_float4(a[0].x, a[0].y, a[1].x, a[1].y);
            reinterpret_cast<float4*>(aip + v)[1] = make_float4(a[2].x, a[2].y, a[3].x, a[3].y);
        } else {
            aip[v] = a[0];
        }
    } else if constexpr (kV == 4) {
        store4<true>(dsrc + v, acc);
    } else {
        dsrc[v] = acc[0];
    }
}

__device__ __forceinline__ float sigmoidf_(float x) { return 1.0f / (1.0f + expf(-x)); }

__device__ __forceinline__ unsigned fast_div(unsigned n, FastDiv f) {
    const unsigned t = __umulhi(f.m, n);
    return (t + ((n - t) >> f.s1)) >> f.s2;
}


}  // namespace gs
#endif

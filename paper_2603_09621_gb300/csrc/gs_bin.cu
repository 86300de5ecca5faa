// gs_bin.cu -- Sec. 3.3 brick intersection and binning: per-Gaussian activation and bounds,
// per-brick Gaussian lists built by count / exclusive scan / stable radix scatter.
//
// Pipeline of gs_bin_bricks (all asynchronous on one stream):
//   k_preprocess    one thread per Gaussian: validity, FP32 brick range (fixed operation order,
//                   bit-exact against the oracle's binning specification), render record. A block
//                   also counts the pairs of its tile of 64 or 256 Gaussians and their first digits.
//   k_row_scan      one block per digit: exclusive scan of the digit's counts over the Gaussian
//                   tiles; one more block scans the tiles' pair counts, stores d_npairs and the
//                   status word (GS_STATUS_NONFINITE, GS_STATUS_CAPACITY).
//   k_radix_scatter (first pass) a block writes gm_off of its Gaussians, emits their pairs into
//                   shared memory and scatters them by digit: the Gaussian-major pair list never
//                   goes to memory. Tiles of very many pairs are shared out in parts (first_part).
//   later passes    the same scan and scatter over tiles of 2,048 pairs, whose digit counts the
//                   scatter before added up or, for large clouds, k_tile_count counts. Stability
//                   keeps ascending Gaussian ids inside each brick, so the lists are deterministic.
//                   The last pass stores pair_brick (key), pair_gmj (Gaussian-major position) and
//                   pair_gid directly.
//   k_brick_off     brick_off from the boundaries of the sorted keys.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#include "gs_common.cuh"

namespace gs {

// ============================================================================ validation

gs_status validate_grid_cfg(const gs_grid* g, const gs_config* c) {
    if (!g || !c) return GS_ERR_INVALID_ARG;
    if (g->nx <= 0 || g->ny <= 0 || g->nz <= 0) return GS_ERR_INVALID_ARG;
    if (int64_t(g->nx) * g->ny * g->nz > (int64_t(1) << 31) - 1) return GS_ERR_INVALID_ARG;
    for (int k = 0; k < 3; ++k) {
        if (!(g->h[k] > 0.0f) || !isfinite(g->h[k]) || !isfinite(g->origin[k]))
            return GS_ERR_INVALID_ARG;
        if (c->brick[k] <= 0 || c->brick[k] % 4 != 0) return GS_ERR_INVALID_ARG;
    }
    // rows of bx voxels along x (bx in {4, 8, 16}), at most 64 rows per brick
    if (c->brick[0] != 4 && c->brick[0] != 8 && c->brick[0] != 16) return GS_ERR_INVALID_ARG;
    if (c->brick[1] != 4 && c->brick[1] != 8 && c->brick[1] != 16) return GS_ERR_INVALID_ARG;
    if (c->brick[1] * c->brick[2] > 64) return GS_ERR_INVALID_ARG;
    if (c->brick[0] * c->brick[1] * c->brick[2] > 512) return GS_ERR_INVALID_ARG;
    if (!(c->trunc_sigma > 0.0f) || !isfinite(c->trunc_sigma)) return GS_ERR_INVALID_ARG;
    if (!(c->eps > 0.0f)) return GS_ERR_INVALID_ARG;
    if (c->signal_mode != 0 && c->signal_mode != 1) return GS_ERR_INVALID_ARG;
    if ((c->a_act != 0 && c->a_act != 1) || (c->t_act != 0 && c->t_act != 1))
        return GS_ERR_INVALID_ARG;
    BrickGeom b = brick_geom(g, c);
    if (int64_t(b.nbx) * b.nby * b.nbz > (int64_t(1) << 30)) return GS_ERR_INVALID_ARG;
    return GS_OK;
}

// ============================================================================ scan

template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Block-wide exclusive scan of one value per thread; returns the exclusive prefix and the
// block total. smem must hold 32 values. Ends with a barrier (smem reusable afterwards).
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* smem, T* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    T inc = warp_inclusive_scan(v, lane);
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T s = lane < nwarps ? smem[lane] : T(0);
        s = warp_inclusive_scan(s, lane);
        smem[lane] = s;
    }
    __syncthreads();
    T prefix = (warp > 0 ? smem[warp - 1] : T(0)) + inc - v;
    *total = smem[nwarps - 1];
    __syncthreads();
    return prefix;
}

// ============================================================================ preprocess

struct GridF {
    int n[3];
    float h[3];
    float o[3];
    float ih[3];  // 1 / h
    int b[3];
    int nb[3];
    FastDiv db[3];  // division by the brick size along each axis
    bool pow2[3];   // h is a power of two (and ih finite and exact): x / h and x ih round alike
};

// x / h_k correctly rounded.
__device__ __forceinline__ float div_h(float x, const GridF& G, int k) {
    return G.pow2[k] ? __fmul_rn(x, G.ih[k]) : __fdiv_rn(x, G.h[k]);
}

// Error-free sum (Knuth): s + e == a + b exactly, s = fl(a + b).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Box of bricks of one Gaussian: first brick and size along each axis; cnt = 0: no brick.
struct BrickBox {
    int lo[3], n[3];
    int cnt;
};

// Key of the box's j-th brick (x fastest).
__device__ __forceinline__ int box_key(const BrickBox& B, int j, int nbx, int nby) {
    const int r = j / B.n[0], x = j - r * B.n[0];
    const int z = r / B.n[1], y = r - z * B.n[1];
    return ((B.lo[2] + z) * nby + B.lo[1] + y) * nbx + B.lo[0] + x;
}

__device__ __forceinline__ BrickBox box_of_lane(const BrickBox& B, int src) {
    BrickBox o;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o.lo[k] = __shfl_sync(0xffffffffu, B.lo[k], src);
        o.n[k] = __shfl_sync(0xffffffffu, B.n[k], src);
    }
    o.cnt = __shfl_sync(0xffffffffu, B.cnt, src);
    return o;
}

// f(source lane, off + j, key) for the bricks j in [j0, j1) of each lane's box. A lane walks up to
// kBoxSerial bricks itself; longer ranges (a Gaussian across much of the volume) are shared by
// the warp. All lanes of the warp call it, lanes without bricks with j0 >= j1.
constexpr int kBoxSerial = 64;

template <typename F>
__device__ __forceinline__ void for_box(const BrickBox& B, int j0, int j1, int off, int nbx, int nby, F f) {
    const int lane = threadIdx.x & 31;
    unsigned big = __ballot_sync(0xffffffffu, j1 - j0 > kBoxSerial);
    if (j1 > j0 && j1 - j0 <= kBoxSerial) {
        int x = 0, y = 0, z = 0;
        if (j0 > 0) {
            const int r = j0 / B.n[0];
            x = j0 - r * B.n[0];
            z = r / B.n[1];
            y = r - z * B.n[1];
        }
        int key = ((B.lo[2] + z) * nby + B.lo[1] + y) * nbx + B.lo[0] + x;
        const int next_row = nbx - B.n[0], next_plane = (nby - B.n[1]) * nbx;
        for (int j = j0; j < j1; ++j) {
            f(lane, off + j, key);
            ++key;
            if (++x == B.n[0]) {
                x = 0;
                key += next_row;
                if (++y == B.n[1]) {
                    y = 0;
                    key += next_plane;
                }
            }
        }
    }
    while (big) {
        const int src = __ffs(big) - 1;
        big &= big - 1;
        const BrickBox o = box_of_lane(B, src);
        const int a = __shfl_sync(0xffffffffu, j0, src), e = __shfl_sync(0xffffffffu, j1, src);
        const int so = __shfl_sync(0xffffffffu, off, src);
        for (int j = a + lane; j < e; j += 32) f(src, so + j, box_key(o, j, nbx, nby));
    }
}

// Range, record and brick box of Gaussian g; returns false where it is invalid (then it has no
// brick and a zero record).
__device__ __forceinline__ bool preprocess_one(const float* __restrict__ params, int64_t g, const GridF& G,
                                               float trunc_sigma, int signal_mode, int a_act, int t_act,
                                               float* __restrict__ rec, int32_t* __restrict__ brange,
                                               BrickBox& box) {
    const float4* p4 = reinterpret_cast<const float4*>(params + g * 12);
    float4 a0 = p4[0], a1 = p4[1], a2 = p4[2];
    float p[12] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w, a2.x, a2.y, a2.z, a2.w};
    int32_t* br = brange + g * 8;
    float4* r4 = reinterpret_cast<float4*>(rec + g * REC_FLOATS);

    bool ok = true;
#pragma unroll
    for (int k = 0; k < 12; ++k) ok = ok && isfinite(p[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) ok = ok && (fabsf(p[3 + k]) <= 30.0f);
    float nn = __fmul_rn(p[6], p[6]);
    nn = __fadd_rn(nn, __fmul_rn(p[7], p[7]));
    nn = __fadd_rn(nn, __fmul_rn(p[8], p[8]));
    nn = __fadd_rn(nn, __fmul_rn(p[9], p[9]));
    ok = ok && (nn > 0.0f);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!ok) {
#pragma unroll
        for (int k = 0; k < 8; ++k) br[k] = 0;
#pragma unroll
        for (int k = 0; k < REC_F4; ++k) r4[k] = z4;
        return false;
    }

    // ---- binning specification (FP32, explicit rounding, fixed order) ----
    float s[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k] = exp_cw(p[3 + k]);
    const float n = __fsqrt_rn(nn);
    const float w = __fdiv_rn(p[6], n), x = __fdiv_rn(p[7], n);
    const float y = __fdiv_rn(p[8], n), z = __fdiv_rn(p[9], n);
    const float xx = __fmul_rn(x, x), yy = __fmul_rn(y, y), zz = __fmul_rn(z, z);
    const float xy = __fmul_rn(x, y), xz = __fmul_rn(x, z), yz = __fmul_rn(y, z);
    const float wx = __fmul_rn(w, x), wy = __fmul_rn(w, y), wz = __fmul_rn(w, z);
    float R[3][3];
    R[0][0] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(yy, zz)));
    R[0][1] = __fmul_rn(2.0f, __fsub_rn(xy, wz));
    R[0][2] = __fmul_rn(2.0f, __fadd_rn(xz, wy));
    R[1][0] = __fmul_rn(2.0f, __fadd_rn(xy, wz));
    R[1][1] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(xx, zz)));
    R[1][2] = __fmul_rn(2.0f, __fsub_rn(yz, wx));
    R[2][0] = __fmul_rn(2.0f, __fsub_rn(xz, wy));
    R[2][1] = __fmul_rn(2.0f, __fadd_rn(yz, wx));
    R[2][2] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(xx, yy)));
    const float ksig = __fmul_rn(trunc_sigma, 1.0001220703125f);
    float sd[3];  // standard deviations along the axes
    int lo[3], hi[3];
    bool inside = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float m0 = __fmul_rn(R[k][0], s[0]), m1 = __fmul_rn(R[k][1], s[1]);
        float m2 = __fmul_rn(R[k][2], s[2]);
        float sig = __fmul_rn(m0, m0);
        sig = __fadd_rn(sig, __fmul_rn(m1, m1));
        sig = __fadd_rn(sig, __fmul_rn(m2, m2));
        sd[k] = __fsqrt_rn(sig);
        float e = __fmul_rn(ksig, sd[k]);
        float lo_f = __fsub_rn(__fsub_rn(div_h(__fsub_rn(__fsub_rn(p[k], e), G.o[k]), G, k), 0.5f), 0.00390625f);
        float hi_f = __fadd_rn(__fsub_rn(div_h(__fsub_rn(__fadd_rn(p[k], e), G.o[k]), G, k), 0.5f), 0.00390625f);
        float nmax = static_cast<float>(G.n[k] - 1);
        if (!(hi_f >= 0.0f) || !(lo_f <= nmax)) {
            inside = false;
        } else {
            float lc = ceilf(lo_f), hc = floorf(hi_f);
            lc = fmaxf(lc, 0.0f);
            hc = fminf(hc, nmax);
            if (lc > hc) inside = false;
            lo[k] = static_cast<int>(lc);
            hi[k] = static_cast<int>(hc);
        }
    }
    if (inside) {
        int b0[3], b1[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            b0[k] = static_cast<int>(fast_div(static_cast<unsigned>(lo[k]), G.db[k]));
            b1[k] = static_cast<int>(fast_div(static_cast<unsigned>(hi[k]), G.db[k]));
            box.lo[k] = b0[k];
            box.n[k] = b1[k] - b0[k] + 1;
        }
        box.cnt = box.n[0] * box.n[1] * box.n[2];
        reinterpret_cast<int4*>(br)[0] = make_int4(b0[0], b0[1], b0[2], b1[0]);
        reinterpret_cast<int4*>(br)[1] = make_int4(b1[1], b1[2], box.cnt, 1);
    } else {
        reinterpret_cast<int4*>(br)[0] = make_int4(0, 0, 0, 0);
        reinterpret_cast<int4*>(br)[1] = make_int4(0, 0, 0, 1);
    }

    // ---- render record (accuracy only; contraction allowed) ----
    // M = sqrt(log2 e / 2) diag(1/s) R^T H: row k of M is R[:, k]^T H scaled by sqrt(k)/s_k.
    const float sk = 0.8493218002880191f;  // sqrt((1/2) log2 e)
    float Mx[3][3];                        // Mx[row][col]
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float f = sk / s[k];
#pragma unroll
        for (int j = 0; j < 3; ++j) Mx[k][j] = f * R[j][k] * G.h[j];
    }
    float col[3][3];  // col[j] = column j of M
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) col[j][k] = Mx[k][j];
    const float am0 = col[0][0] * col[0][0] + col[0][1] * col[0][1] + col[0][2] * col[0][2];
    const float inv_a = 1.0f / am0;
    float nrm[3];
#pragma unroll
    for (int j = 0; j < 3; ++j)
        nrm[j] = sqrtf(col[j][0] * col[j][0] + col[j][1] * col[j][1] + col[j][2] * col[j][2]);
    // n1, n2: m1, m2 with their components along m0 removed; c_j = -(m_j . m0) / a
    float n1[3], n2[3];
    const float d1 = (col[1][0] * col[0][0] + col[1][1] * col[0][1] + col[1][2] * col[0][2]) * inv_a;
    const float d2 = (col[2][0] * col[0][0] + col[2][1] * col[0][1] + col[2][2] * col[0][2]) * inv_a;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        n1[k] = col[1][k] - d1 * col[0][k];
        n2[k] = col[2][k] - d2 * col[0][k];
    }
    const float Pyy = n1[0] * n1[0] + n1[1] * n1[1] + n1[2] * n1[2];
    const float Pzz = n2[0] * n2[0] + n2[1] * n2[1] + n2[2] * n2[2];
    const float P2yz = 2.0f * (n1[0] * n2[0] + n1[1] * n2[1] + n1[2] * n2[2]);
    // Mean in voxel-index space m = (mu - o) / h - 1/2 as a float head + tail, in double-float
    // arithmetic (Knuth's error-free two-sum; the quotient's remainder from one FMA), so that
    // m = mh + ml to about 2^-46 relative and d = (i - mh) - ml keeps one rounding at any
    // coordinate. (FP64 runs at 1/64 of the FP32 rate here.)
    float mh[3], ml[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float dh, dl;
        two_sum(p[k], -G.o[k], dh, dl);           // mu - o exactly
        const float qh = div_h(dh, G, k);         // correctly rounded: the remainder is exact
        const float rem = fmaf(-qh, G.h[k], dh);
        const float ql = __fmul_rn(__fadd_rn(rem, dl), G.ih[k]);
        float sh, sl;
        two_sum(qh, -0.5f, sh, sl);
        two_sum(sh, __fadd_rn(sl, ql), mh[k], ml[k]);
    }
    float A = a_act ? sigmoidf_(p[10]) : p[10];
    float T = t_act ? sigmoidf_(p[11]) : p[11];
    float v, r;
    if (signal_mode == 0) {
        v = A;
        r = T;
    } else {
        v = A * T;
        r = 1.0f;
    }
    r4[0] = make_float4(-mh[0], -ml[0], -mh[1], -mh[2]);
    r4[1] = make_float4(-ml[1], -ml[2], P2yz, -d2);
    r4[2] = make_float4(Pyy, -d1, Pzz, nrm[0]);
    // radius of a 4^3 footprint in whitened units: |M d|^2 <= sum_jk |m_j . m_k| (3/2)^2
    float gsum = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            gsum += fabsf(col[j][0] * col[k][0] + col[j][1] * col[k][1] + col[j][2] * col[k][2]);
    const float rho4 = 1.5f * sqrtf(gsum);
    // half-extents of the truncated ellipsoid's box in voxels, widened by 1 % and by a 4^3
    // footprint's half-width: a footprint whose centre is farther along an axis is missed
    float ext[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ext[k] = 1.01f * trunc_sigma * sd[k] * G.ih[k] + 1.5f + 1e-3f;
    r4[3] = make_float4(ext[0], rho4, ext[1], ext[2]);
    // lower bound of q per squared voxel distance from the mean: (log2 e / 2) h_min^2 / s_max^2
    // bounds the smallest eigenvalue of the voxel-space form (less 1e-3 for rounding), so
    // a footprint whose voxel box lies farther than sqrt(Tcull / lam) from the mean is missed
    const float smax = fmaxf(s[0], fmaxf(s[1], s[2]));
    const float hmin = fminf(G.h[0], fminf(G.h[1], G.h[2]));
    const float lam = kHalfLog2e * (1.0f - 1e-3f) * (hmin / smax) * (hmin / smax);
    r4[4] = make_float4(v * r, r, v, lam);
    return true;
}

// Digit counts of `len` pairs of consecutive keys from `key` on (a row of a box): a constant on all
// digits, added to hall, and 1 on an interval of digits, as differences in hdif.
__device__ __forceinline__ void count_row(int key, int len, int nd, int* hdif, int* hall) {
    const int a = key & (nd - 1);
    const int rem = len & (nd - 1), e = a + rem;
    if (len >= nd) atomicAdd(hall, len / nd);
    if (rem) {
        atomicAdd(&hdif[a], 1);
        if (e <= nd) {
            atomicAdd(&hdif[e], -1);
        } else {
            atomicAdd(&hdif[0], 1);
            atomicAdd(&hdif[e - nd], -1);
        }
    }
}

constexpr long long kBadFlag = 1LL << 62;  // marks a Gaussian tile with an invalid Gaussian

// Six blocks of 256 per SM (42 registers, a few values spilled to L1) measured faster than
// four (52 registers, no spills): the kernel is latency-bound on its division and square-root
// sequences, so the extra resident warps pay more than the spills cost. Where the voxel size is a
// power of two (unit spacing above all) nine of its seventeen divisions are exact products: 23.4 -> 22.2
// us at 500,000 Gaussians.
// The block also stores its column of the first radix pass's digit counts (hist0[d * stride0 +
// block]) and its number of pairs (blk[block]), kBadFlag added where a Gaussian was invalid.
template <int kTile>
__global__ void __launch_bounds__(kTile, 6 * 256 / kTile) k_preprocess(
    const float* __restrict__ params, int64_t N, GridF G, float trunc_sigma, int signal_mode, int a_act,
    int t_act, float* __restrict__ rec, int32_t* __restrict__ brange, int nd, int32_t* __restrict__ hist0,
    int64_t stride0, long long* __restrict__ blk) {
    pdl_enter();
    static_assert((kTile & (kTile - 1)) == 0, "the digits (a power of two) divide evenly among the threads");
    __shared__ int hcnt[kMaxDigits], hdif[kMaxDigits + 1], sscan[32];
    __shared__ int hall, flags;  // flags: 1 an invalid Gaussian, 2 a box of more than kBoxSerial bricks
    __shared__ unsigned long long btot;
    for (int d = threadIdx.x; d <= nd; d += kTile) {
        if (d < nd) hcnt[d] = 0;
        hdif[d] = 0;
    }
    if (threadIdx.x == 0) {
        hall = flags = 0;
        btot = 0;
    }
    __syncthreads();
    const int64_t g = int64_t(blockIdx.x) * kTile + threadIdx.x;
    BrickBox box;
    box.cnt = 0;
    bool bad = false;
    if (g < N)
        bad = !preprocess_one(params, g, G, trunc_sigma, signal_mode, a_act, t_act, rec, brange, box);
    unsigned long long wsum = static_cast<unsigned>(box.cnt);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
    const int lane = threadIdx.x & 31;
    if (lane == 0 && wsum != 0) atomicAdd(&btot, wsum);
    for_box(box, 0, box.cnt <= kBoxSerial ? box.cnt : 0, 0, G.nb[0], G.nb[1],
            [&](int, int, int key) { atomicAdd(&hcnt[key & (nd - 1)], 1); });
    // larger boxes by rows of consecutive keys, shared by the warp: a row adds a constant to every
    // digit and 1 to an interval of digits (as differences), so that a cloud whose pairs will
    // exceed the capacity costs no more than its rows
    unsigned big = __ballot_sync(0xffffffffu, box.cnt > kBoxSerial);
    const int warp_flags = (__any_sync(0xffffffffu, bad) ? 1 : 0) | (big != 0 ? 2 : 0);
    if (lane == 0 && warp_flags != 0) atomicOr(&flags, warp_flags);
    while (big) {
        const int src = __ffs(big) - 1;
        big &= big - 1;
        const BrickBox o = box_of_lane(box, src);
        for (int r = lane; r < o.n[1] * o.n[2]; r += 32) {
            const int z = r / o.n[1], y = r - z * o.n[1];
            count_row(((o.lo[2] + z) * G.nb[1] + o.lo[1] + y) * G.nb[0] + o.lo[0], o.n[0], nd, hdif, &hall);
        }
    }
    __syncthreads();
    const int di = nd > kTile ? nd / kTile : 1;  // thread t stores digits [t di, (t + 1) di)
    int run = 0;
    if (flags & 2) {
        int v = 0, tot;
        for (int e = 0; e < di; ++e) v += threadIdx.x * di + e < nd ? hdif[threadIdx.x * di + e] : 0;
        run = block_exclusive_scan(v, sscan, &tot) + hall;
    }
    for (int e = 0; e < di; ++e) {
        const int d = threadIdx.x * di + e;
        if (d < nd) {
            if (flags & 2) run += hdif[d];
            hist0[d * stride0 + blockIdx.x] = hcnt[d] + run;
        }
    }
    if (threadIdx.x == 0) blk[blockIdx.x] = static_cast<long long>(btot) + ((flags & 1) ? kBadFlag : 0);
}

// ============================================================================ radix sort

__device__ __forceinline__ int64_t valid_pairs(const int64_t* npairs, int64_t capacity) {
    int64_t P = *npairs;
    return (P > capacity || P < 0) ? 0 : P;
}

constexpr int kRowThreads = 512;
constexpr int kRowItems = 4;

struct RowScan {
    int32_t* hist;       // rows of digit counts, scanned in place (exclusive within a row)
    int64_t stride;
    int64_t cols;        // columns in use: fixed (first pass), or from npairs where < 0
    int32_t* rowtot;     // row totals
    int32_t* zero;       // the next pass's counts, cleared here where the scatter adds them up (else nullptr)
    int zero_rows;
    int64_t zero_stride;
    long long* blk;      // first pass: pairs of each Gaussian tile, scanned by the last block,
    int32_t* ticket;     // which also clears the loss kernel's block counter
    int nd;
    int64_t* npairs;
    int64_t capacity;
    int32_t* status;
};

// Block d scans row d (digit d's counts over the tiles) and clears the next pass's counts where these are
// added up by atomics; the scatter adds up the row totals before its digits itself, so a pass's scan is one
// launch of 3.5 us at 1,954 tiles (a reduction and a down-sweep over all rows took two, 9 us).
// The first pass's block nd scans the Gaussian tiles' pair counts (64-bit).
__global__ void __launch_bounds__(kRowThreads) k_row_scan(RowScan A) {
    pdl_enter();
    __shared__ long long sm[32];
    const int row = blockIdx.x, tid = threadIdx.x;
    long long carry = 0;
    if (row == A.nd) {
        __shared__ int bad;
        __shared__ long long heaviest;
        if (tid == 0) {
            bad = 0;
            heaviest = 0;
        }
        __syncthreads();
        long long most = 0;
        for (int64_t c0 = 0; c0 < A.cols; c0 += kRowThreads) {
            const int64_t c = c0 + tid;
            long long v = c < A.cols ? A.blk[c] : 0;
            if (v >= kBadFlag) {
                v -= kBadFlag;
                bad = 1;
            }
            most = v > most ? v : most;
            long long tot;
            const long long pre = block_exclusive_scan(v, sm, &tot);
            if (c < A.cols) A.blk[c] = carry + pre;
            carry += tot;
        }
        if (most > kFirstMinPart) atomicMax(&heaviest, most);
        __syncthreads();
        if (tid == 0) {
            A.blk[A.cols] = carry;
            A.blk[A.cols + 1] = heaviest;
            *A.ticket = 0;
            *A.npairs = carry;
            *A.status = (bad ? GS_STATUS_NONFINITE : 0) | (carry > A.capacity ? GS_STATUS_CAPACITY : 0);
        }
        return;
    }
    const int64_t cols = A.cols >= 0 ? A.cols : (valid_pairs(A.npairs, A.capacity) + kSortTile - 1) / kSortTile;
    int32_t* h = A.hist + row * A.stride;
    for (int64_t c0 = 0; c0 < cols; c0 += kRowThreads * kRowItems) {
        const int64_t c = c0 + int64_t(tid) * kRowItems;
        // (the stride is a multiple of 4, so a 16-byte piece that starts inside the row is whole)
        int4 v = c < cols ? *reinterpret_cast<const int4*>(h + c) : make_int4(0, 0, 0, 0);
        if (c + 1 >= cols) v.y = 0;
        if (c + 2 >= cols) v.z = 0;
        if (c + 3 >= cols) v.w = 0;
        long long tot;
        const int s = v.x + v.y + v.z + v.w;
        const int pre = static_cast<int>(carry + block_exclusive_scan<long long>(s, sm, &tot));
        if (c < cols)
            *reinterpret_cast<int4*>(h + c) = make_int4(pre, pre + v.x, pre + v.x + v.y, pre + v.x + v.y + v.z);
        carry += tot;
    }
    if (tid == 0) A.rowtot[row] = static_cast<int>(carry);
    if (A.zero)
        for (int r = row; r < A.zero_rows; r += A.nd)
            for (int64_t c = int64_t(tid) * 4; c < A.zero_stride; c += kRowThreads * 4)
                *reinterpret_cast<int4*>(A.zero + r * A.zero_stride + c) = make_int4(0, 0, 0, 0);
}

// Digit counts of a later pass, a column per tile of kSortTile pairs of the pass before: a block counts
// kCountTiles tiles in shared memory and writes their columns in 16-byte pieces. Bound by the keys' read.
constexpr int kCountTiles = 4;

__global__ void __launch_bounds__(kSortThreads) k_tile_count(const int32_t* __restrict__ keys,
                                                             const int64_t* __restrict__ npairs, int64_t capacity,
                                                             int shift, int nd, int32_t* __restrict__ hist,
                                                             int64_t stride) {
    pdl_enter();
    __shared__ int cnt[kCountTiles][kMaxDigits];
    const int64_t P = valid_pairs(npairs, capacity);
    const int64_t tile0 = int64_t(blockIdx.x) * kCountTiles;
    if (tile0 * kSortTile >= P) return;
    for (int d = threadIdx.x; d < nd; d += kSortThreads)
#pragma unroll
        for (int t = 0; t < kCountTiles; ++t) cnt[t][d] = 0;
    __syncthreads();
    constexpr int kPieces = kSortTile / (4 * kSortThreads);  // of 16 bytes per thread and tile
    int4 k[kCountTiles * kPieces];
#pragma unroll
    for (int e = 0; e < kCountTiles * kPieces; ++e) {
        const int64_t i = tile0 * kSortTile + (e * kSortThreads + threadIdx.x) * 4;
        k[e] = make_int4(-1, -1, -1, -1);
        if (i + 3 < P) {
            k[e] = *reinterpret_cast<const int4*>(keys + i);
        } else {
            if (i < P) k[e].x = keys[i];
            if (i + 1 < P) k[e].y = keys[i + 1];
            if (i + 2 < P) k[e].z = keys[i + 2];
        }
    }
#pragma unroll
    for (int e = 0; e < kCountTiles * kPieces; ++e) {
        int* c = cnt[e / kPieces];
        if (k[e].x >= 0) atomicAdd(&c[(k[e].x >> shift) & (nd - 1)], 1);
        if (k[e].y >= 0) atomicAdd(&c[(k[e].y >> shift) & (nd - 1)], 1);
        if (k[e].z >= 0) atomicAdd(&c[(k[e].z >> shift) & (nd - 1)], 1);
        if (k[e].w >= 0) atomicAdd(&c[(k[e].w >> shift) & (nd - 1)], 1);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nd; d += kSortThreads)
        *reinterpret_cast<int4*>(hist + d * stride + tile0) = make_int4(cnt[0][d], cnt[1][d], cnt[2][d], cnt[3][d]);
}

struct Scatter {
    const int32_t* keys_in;    // pass input (not the first pass)
    const int2* vals_in;       // (Gaussian-major position, Gaussian id)
    int32_t* keys_out;         // the last pass: pair_brick
    int2* vals_out;            // (not the last pass)
    int32_t* out_gmj;          // last pass
    int32_t* out_gid;
    const int32_t* hist;       // this pass's scanned counts
    int64_t stride;
    const int32_t* rowtot;
    int32_t* hist_next;        // the next pass's counts where this one adds them up (else nullptr)
    int64_t stride_next;
    int bits_next;
    int shift, bits;
    const int64_t* npairs;
    int64_t capacity;
    const int32_t* brange;     // first pass: emission
    int32_t* gm_off;
    const long long* blk_base;
    int64_t N;
    int nbx, nby;
    int nb;                    // bricks
    int32_t* brick_off;        // (a first pass that is the last)
    unsigned tiles;            // first pass: blocks from this one on take parts of the heavy tiles
    unsigned block0;           // and the grid's first block
};

// Stable scatter of one tile of up to kRound keys per round. Warp w owns a contiguous part of the tile
// and visits it in rounds of 32 consecutive keys, kept in registers with their ranks among the warp's
// earlier equal digits (warp match masks). A block-wide prefix over the digits then gives each digit's
// run inside the tile and each warp's start in it; the tile is placed in shared memory sorted by digit,
// ties in tile order, and written out in that order, so consecutive threads store consecutive addresses
// of a run.
// kFirst: the tile is emitted by the block itself from its kTile Gaussians' boxes (in rounds of kRound
// pairs; the digits' output positions advance from round to round; what a tile has beyond first_part
// pairs is left to blocks for parts, whose rounds start further on: 64 Gaussians on 16,384 bricks, 1.05M
// pairs in one tile, 6.35 -> 0.17 ms, on 131,072 bricks 51.4 -> 0.7 ms), else it is one tile of the
// previous pass's output. kLast: the pass stores the bins' per-pair arrays; every other pass of a small
// cloud adds each key to the next pass's digit counts at its output position's tile (one atomic per group
// of equal (tile, digit) in a warp).
// Bound by latency (barriers, the gathered loads) at 40-65 % issue-active, far from bandwidth: the pair
// list is cache-resident at the fitting size. Whole binning, L2 flushed, at 3.26M pairs (256 x 256 x 128
// grid, 8^3 bricks): 115 us with the pair list emitted to memory, two scan launches per list and the
// owners gathered in the last pass; 88 us now (preprocess 22, first pass 28, last pass 20, count 4, scans
// 7, offsets 6). 104M pairs (512 x 512 x 256, digits of 9 and 8 bits where 8-bit digits took three
// passes): 5.86 -> 2.36 ms. 21,828 pairs (32^3): 30 -> 17 us. At 3.26M pairs: ranks recomputed by a
// second match per key and the values held in registers (80 registers) 108 us; the values loaded when the
// tile is placed 0.17 ms longer at 104M than copied to shared memory asynchronously during the ranking
// (here); 5 (6) blocks per SM with spills 95 (97) us.
template <bool kFirst, bool kLast, int kTile>
__global__ void __launch_bounds__(kSortThreads, 4) k_radix_scatter(Scatter A) {
    pdl_enter();
    constexpr int kWarps = kSortThreads / 32;
    static_assert(kSortThreads >= kTile, "one thread per Gaussian of a tile");
    constexpr int kMaxRound = kSortThreads * (kFirst ? kFirstItems : kSortItems);
    static_assert(kMaxRound < 8192, "runs of a round are packed in 13 bits");
    const int nd = 1 << A.bits, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    extern __shared__ int smem[];
    int* wcnt = smem;                 // [kWarps][nd]
    int* goff = wcnt + kWarps * nd;   // output position of tile slot j of digit d: goff[d] + j
    __shared__ __align__(16) int skey[kMaxRound];
    __shared__ unsigned short sidx[kMaxRound];             // sorted: tile index of each key
    __shared__ unsigned char sowner[kFirst ? kMaxRound : 1];  // tile order: Gaussian of the block
    __shared__ int2 sval[kFirst ? 1 : kSortTile];       // tile order: the keys' values
    __shared__ long long sscan[32];

    const int64_t P = valid_pairs(A.npairs, A.capacity);
    int64_t base = int64_t(blockIdx.x) * kSortTile;  // first pair (Gaussian-major in the first pass)
    int tile = kFirst ? blockIdx.x + A.block0 : blockIdx.x;
    int begin = 0, end;                              // pairs of the tile that this block places
    BrickBox box;
    box.cnt = 0;
    int loc = 0;                                     // the thread's first pair in the block
    int gpos[kMaxDigits / kSortThreads] = {};        // the thread's digits' next output positions (first: what
                                                     // the tile places before `begin`)
    if (kFirst) {
        const int64_t part = first_part(P);
        const bool own = static_cast<unsigned>(tile) < A.tiles;
        if (!own) {
            // the part [p0, p0 + part) of the pair list, as far as it lies behind the first `part` pairs
            // of the tile that p0 falls in (any later tile's share of it is its own block's)
            const int64_t p0 = int64_t(tile - A.tiles) * part;
            if (A.blk_base[A.tiles + 1] <= part || p0 >= P) return;
            int hi = static_cast<int>(A.tiles) - 1;
            for (tile = 0; tile < hi;) {
                const int mid = (tile + hi + 1) >> 1;
                if (A.blk_base[mid] <= p0)
                    tile = mid;
                else
                    hi = mid - 1;
            }
            const int64_t b = A.blk_base[tile], n = A.blk_base[tile + 1] - b;
            begin = static_cast<int>(max(p0 - b, part));
            end = static_cast<int>(min(p0 + part - b, n));
            if (begin >= end) return;
        }
        const int64_t g = tid < kTile ? int64_t(tile) * kTile + tid : A.N;
        if (g < A.N) {
            const int4 lo = reinterpret_cast<const int4*>(A.brange + g * 8)[0];
            const int4 hi = reinterpret_cast<const int4*>(A.brange + g * 8)[1];
            box.lo[0] = lo.x; box.lo[1] = lo.y; box.lo[2] = lo.z;
            box.n[0] = lo.w - lo.x + 1; box.n[1] = hi.x - lo.y + 1; box.n[2] = hi.y - lo.z + 1;
            box.cnt = hi.z;
        }
        base = A.blk_base[tile];
        // (offsets modulo 2^32: exact where the pairs fit the capacity, which is below 2^31)
        unsigned tot;
        const unsigned pre = block_exclusive_scan(static_cast<unsigned>(box.cnt),
                                                  reinterpret_cast<unsigned*>(sscan), &tot);
        if (own && g < A.N) {
            A.gm_off[g] = static_cast<int32_t>(static_cast<unsigned>(base) + pre);
            if (g == A.N - 1) A.gm_off[A.N] = static_cast<int32_t>(static_cast<unsigned>(base) + pre + box.cnt);
        }
        if (kLast && blockIdx.x + A.block0 == 0) {
            // the only pass: a digit is a brick, so the digits' exclusive prefix is brick_off
            const int di = nd > kSortThreads ? nd / kSortThreads : 1;
            int row[kMaxDigits / kSortThreads], mine = 0, all;
#pragma unroll
            for (int e = 0; e < kMaxDigits / kSortThreads; ++e) {
                const int d = tid * di + e;
                row[e] = (P > 0 && e < di && d < nd) ? A.rowtot[d] : 0;
                mine += row[e];
            }
            int run = block_exclusive_scan(mine, reinterpret_cast<int*>(sscan), &all);
#pragma unroll
            for (int e = 0; e < kMaxDigits / kSortThreads; ++e) {
                const int d = tid * di + e;
                if (e < di && d <= A.nb) A.brick_off[d] = run;
                run += row[e];
            }
            if (tid == 0 && A.nb == nd) A.brick_off[nd] = all;
        }
        if (P == 0) return;  // also when the pairs exceed the capacity
        loc = static_cast<int>(pre);
        if (own) {
            end = static_cast<int>(min(int64_t(tot), part));
        } else {
            // digit counts of the tile's pairs before `begin`: its boxes staged in skey (first pair, size
            // along x and y, first key), their rows shared by all warps
            static_assert(kMaxRound >= 4 * kTile, "a tile's boxes fit the key buffer");
            int4* sbox = reinterpret_cast<int4*>(skey);
            int* hdif = wcnt;
            if (tid < kTile)
                sbox[tid] = make_int4(min(max(begin - loc, 0), box.cnt), box.n[0], box.n[1],
                                      (box.lo[2] * A.nby + box.lo[1]) * A.nbx + box.lo[0]);
            for (int d = tid; d <= nd + 1; d += kSortThreads) hdif[d] = 0;
            __syncthreads();
            for (int t = warp; t < kTile; t += kWarps) {
                const int4 b = sbox[t];  // (pairs before `begin`, row length, rows per plane, first key)
                if (b.x == 0) continue;
                for (int r = lane; r <= (b.x - 1) / b.y; r += 32) {
                    const int z = r / b.z, y = r - z * b.z;
                    count_row(b.w + (z * A.nby + y) * A.nbx, min(b.y, b.x - r * b.y), nd, hdif, &hdif[nd + 1]);
                }
            }
            __syncthreads();
            const int di = nd > kSortThreads ? nd / kSortThreads : 1;
            int v = 0, sum;
            for (int e = 0; e < di; ++e) v += tid * di + e < nd ? hdif[tid * di + e] : 0;
            int run = block_exclusive_scan(v, reinterpret_cast<int*>(sscan), &sum) + hdif[nd + 1];
#pragma unroll
            for (int e = 0; e < kMaxDigits / kSortThreads; ++e)
                if (e < di && tid * di + e < nd) gpos[e] = run += hdif[tid * di + e];
            __syncthreads();
        }
    } else {
        if (base >= P) return;  // past the last pair: nothing to place
        end = static_cast<int>(min(int64_t(kSortTile), P - base));
    }
    // rounds of kRound pairs, kItems per thread
    auto rounds_of = [&](auto items) {
        constexpr int kItems = decltype(items)::value, kRound = kSortThreads * kItems;
        for (int c0 = begin; c0 < end; c0 += kRound) {
            const int n = min(kRound, end - c0);
            if (kFirst) {
                if (c0 > begin) __syncthreads();  // the previous round has been written out
                for_box(box, max(0, c0 - loc), min(box.cnt, c0 + n - loc), loc - c0, A.nbx, A.nby,
                        [&](int src, int o, int key) {
                            skey[o] = key;
                            sowner[o] = static_cast<unsigned char>(warp * 32 + src);
                        });
            }
            for (int d = tid; d < kWarps * nd; d += kSortThreads) wcnt[d] = 0;
            __syncthreads();
            // each warp's part: the same number of 32-key rounds
            const int rounds = (n + kSortThreads - 1) / kSortThreads;
            const int sub0 = warp * rounds * 32;
            int kr[kItems];
            unsigned short rank[kItems];
#pragma unroll
            for (int r = 0; r < kItems; ++r) {
                const int idx = sub0 + r * 32 + lane;
                kr[r] = 0;
                if (idx < n && r < rounds) {
                    kr[r] = kFirst ? skey[idx] : A.keys_in[base + idx];
                    if (!kFirst)  // read again only when the sorted tile is written out
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                                         static_cast<unsigned>(__cvta_generic_to_shared(&sval[idx]))),
                                     "l"(A.vals_in + base + idx)
                                     : "memory");
                }
            }
#pragma unroll
            for (int r = 0; r < kItems; ++r) {
                if (r < rounds) {
                    const bool valid = sub0 + r * 32 + lane < n;
                    const int d = (kr[r] >> A.shift) & (nd - 1);
                    const unsigned peers = __match_any_sync(0xffffffffu, valid ? d : nd + lane);
                    int* w = &wcnt[warp * nd + d];
                    const int before = valid ? *w : 0;
                    __syncwarp();
                    if (valid && lane == __ffs(peers) - 1) *w = before + __popc(peers);
                    __syncwarp();
                    rank[r] = static_cast<unsigned short>(before + __popc(peers & ((1u << lane) - 1u)));
                }
            }
            __syncthreads();
            // digit runs: thread t owns digits [t di, (t + 1) di)
            const int di = nd > kSortThreads ? nd / kSortThreads : 1;
            long long mine = 0;
            int runs[kMaxDigits / kSortThreads], rows[kMaxDigits / kSortThreads];
#pragma unroll
            for (int e = 0; e < kMaxDigits / kSortThreads; ++e) {
                runs[e] = rows[e] = 0;
                const int d = tid * di + e;
                if (e < di && d < nd) {
                    int run = 0;
#pragma unroll
                    for (int w = 0; w < kWarps; ++w) {
                        const int c = wcnt[w * nd + d];
                        wcnt[w * nd + d] = run;
                        run += c;
                    }
                    runs[e] = run;
                    if (c0 == begin) rows[e] = A.rowtot[d];
                }
                mine += (static_cast<long long>(rows[e]) << 13) | runs[e];  // (sums of runs: <= kRound)
            }
            long long all;
            const long long pre = block_exclusive_scan(mine, sscan, &all);
            int start = static_cast<int>(pre & 8191);
            int64_t row0 = pre >> 13;
#pragma unroll
            for (int e = 0; e < kMaxDigits / kSortThreads; ++e) {
                const int d = tid * di + e;
                if (e < di && d < nd) {
                    if (c0 == begin) gpos[e] += static_cast<int>(row0) + A.hist[d * A.stride + tile];
                    goff[d] = gpos[e] - start;
                    gpos[e] += runs[e];
#pragma unroll
                    for (int w = 0; w < kWarps; ++w) wcnt[w * nd + d] += start;
                    row0 += rows[e];
                    start += runs[e];
                }
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < kItems; ++r) {
                const int idx = sub0 + r * 32 + lane;
                if (r < rounds && idx < n) {
                    const int lp = wcnt[warp * nd + ((kr[r] >> A.shift) & (nd - 1))] + rank[r];
                    skey[lp] = kr[r];
                    sidx[lp] = static_cast<unsigned short>(idx);
                }
            }
            if (!kFirst) asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            for (int j = tid; j < n; j += kSortThreads) {
                const int key = skey[j];
                const int idx = sidx[j];
                const int2 v = kFirst ? make_int2(static_cast<int>(base) + c0 + idx,
                                                  tile * kTile + sowner[idx])
                                      : sval[idx];
                const int pos = goff[(key >> A.shift) & (nd - 1)] + j;
                A.keys_out[pos] = key;
                if (kLast) {
                    A.out_gmj[pos] = v.x;
                    A.out_gid[pos] = v.y;
                } else {
                    A.vals_out[pos] = v;
                    if (A.hist_next) {
                        const int tile = pos / kSortTile, dn = (key >> (A.shift + A.bits)) & ((1 << A.bits_next) - 1);
                        const unsigned peers = __match_any_sync(__activemask(), (tile << kMaxRadixBits) | dn);
                        if (lane == __ffs(peers) - 1)
                            atomicAdd(&A.hist_next[dn * A.stride_next + tile], __popc(peers));
                    }
                }
            }
        }
    };
    if (kFirst && end - begin > kSortTile)
        rounds_of(std::integral_constant<int, kFirstItems>());
    else
        rounds_of(std::integral_constant<int, kSortItems>());
}

// brick_off from the boundaries of the sorted keys (brick_off[b] = first pair of brick b, or
// the next non-empty brick's first pair; brick_off[nb] = P). Four consecutive keys per thread; runs
// of empty bricks longer than kGapSerial are filled by the whole warp. (One key per thread with
// its predecessor loaded beside it, and gaps filled by one thread, took 600 us at 104M pairs and
// 131,072 bricks.)
constexpr int kGapSerial = 8;

__global__ void __launch_bounds__(256) k_brick_off(const int32_t* __restrict__ keys,
                                                   const int64_t* __restrict__ npairs,
                                                   int64_t capacity, int nb,
                                                   int32_t* __restrict__ brick_off) {
    pdl_enter();
    const int64_t P = valid_pairs(npairs, capacity);
    const int lane = threadIdx.x & 31;
    const int64_t step = int64_t(gridDim.x) * blockDim.x;
    // entry i <= P: key i, and the sentinel key nb at i = P
    for (int64_t q0 = int64_t(blockIdx.x) * blockDim.x + (threadIdx.x & ~31); 4 * q0 <= P; q0 += step) {
        const int64_t i = 4 * (q0 + lane);
        int4 k = make_int4(nb, nb, nb, nb);
        if (i + 3 < P) {
            k = *reinterpret_cast<const int4*>(keys + i);
        } else {
            if (i < P) k.x = keys[i];
            if (i + 1 < P) k.y = keys[i + 1];
            if (i + 2 < P) k.z = keys[i + 2];
        }
        int prev = __shfl_up_sync(0xffffffffu, k.w, 1);
        if (lane == 0) prev = i > 0 ? keys[i - 1] : -1;
        const int cur[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int gap = i + e <= P ? cur[e] - prev : 0;
            if (gap <= kGapSerial)
                for (int b = prev + 1; b <= prev + gap; ++b) brick_off[b] = static_cast<int32_t>(i + e);
            unsigned big = __ballot_sync(0xffffffffu, gap > kGapSerial);
            while (big) {
                const int src = __ffs(big) - 1;
                big &= big - 1;
                const int b0 = __shfl_sync(0xffffffffu, prev, src), g = __shfl_sync(0xffffffffu, gap, src);
                const int v = static_cast<int>(4 * (q0 + src) + e);
                for (int b = lane + 1; b <= g; b += 32) brick_off[b0 + b] = v;
            }
            prev = cur[e];
        }
    }
}

}  // namespace gs

// ============================================================================ C ABI

using namespace gs;

namespace {

struct BinsLayout {
    size_t off_brick_off, off_pair_gid, off_pair_gmj, off_pair_brick, off_gm_off, off_rec, off_brange,
        off_npairs,
        off_status, bytes;
};

bool bins_layout(int64_t n_gauss, int64_t capacity, int32_t n_bricks, BinsLayout* L) {
    if (n_gauss < 0 || capacity < 0 || capacity > kMaxCapacity || n_bricks <= 0) return false;
    if (n_gauss > (int64_t(1) << 31) - 2) return false;
    const int64_t cap = capacity > 0 ? capacity : 1;
    const int64_t n = n_gauss > 0 ? n_gauss : 1;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    L->off_brick_off = take(sizeof(int32_t) * (int64_t(n_bricks) + 1));
    L->off_pair_gid = take(sizeof(int32_t) * cap);
    L->off_pair_gmj = take(sizeof(int32_t) * cap);
    L->off_pair_brick = take(sizeof(int32_t) * cap);
    L->off_gm_off = take(sizeof(int32_t) * (n + 1));
    L->off_rec = take(sizeof(float) * REC_FLOATS * n);
    L->off_brange = take(sizeof(int32_t) * 8 * n);
    L->off_npairs = take(sizeof(int64_t));
    L->off_status = take(sizeof(int32_t));
    L->bytes = off;
    return true;
}

int32_t n_bricks_of(const gs_grid* g, const gs_config* c) {
    BrickGeom b = brick_geom(g, c);
    return b.nbx * b.nby * b.nbz;
}

int64_t n_voxels_of(const gs_grid* g) { return int64_t(g->nx) * g->ny * g->nz; }

}  // namespace

extern "C" size_t gs_bins_bytes(int64_t n_gauss, int64_t capacity, const gs_grid* grid,
                                const gs_config* cfg) {
    if (validate_grid_cfg(grid, cfg) != GS_OK) return 0;
    BinsLayout L;
    if (!bins_layout(n_gauss, capacity, n_bricks_of(grid, cfg), &L)) return 0;
    return L.bytes;
}

extern "C" gs_status gs_bins_bind(void* arena, size_t arena_bytes, int64_t n_gauss,
                                  int64_t capacity, const gs_grid* grid, const gs_config* cfg,
                                  gs_bins* out) {
    if (!arena || !out) return GS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(arena) % 256 != 0) return GS_ERR_INVALID_ARG;
    gs_status s = validate_grid_cfg(grid, cfg);
    if (s != GS_OK) return s;
    BinsLayout L;
    const int32_t nb = n_bricks_of(grid, cfg);
    if (!bins_layout(n_gauss, capacity, nb, &L)) return GS_ERR_INVALID_ARG;
    if (arena_bytes < L.bytes) return GS_ERR_WORKSPACE;
    char* a = static_cast<char*>(arena);
    BrickGeom b = brick_geom(grid, cfg);
    out->n_gauss = n_gauss;
    out->capacity = capacity;
    out->n_bricks = nb;
    out->nbx = b.nbx;
    out->nby = b.nby;
    out->nbz = b.nbz;
    out->brick_off = reinterpret_cast<int32_t*>(a + L.off_brick_off);
    out->pair_gid = reinterpret_cast<int32_t*>(a + L.off_pair_gid);
    out->pair_gmj = reinterpret_cast<int32_t*>(a + L.off_pair_gmj);
    out->pair_brick = reinterpret_cast<int32_t*>(a + L.off_pair_brick);
    out->gm_off = reinterpret_cast<int32_t*>(a + L.off_gm_off);
    out->rec = reinterpret_cast<float*>(a + L.off_rec);
    out->brange = reinterpret_cast<int32_t*>(a + L.off_brange);
    out->d_npairs = reinterpret_cast<int64_t*>(a + L.off_npairs);
    out->d_status = reinterpret_cast<int32_t*>(a + L.off_status);
    return GS_OK;
}

extern "C" size_t gs_workspace_bytes(int64_t n_gauss, int64_t capacity, const gs_grid* grid,
                                     const gs_config* cfg) {
    if (validate_grid_cfg(grid, cfg) != GS_OK) return 0;
    if (n_gauss < 0 || capacity < 0 || capacity > kMaxCapacity) return 0;
    Workspace ws;
    carve_workspace(nullptr, n_gauss, capacity, n_bricks_of(grid, cfg), n_voxels_of(grid),
                    cfg->deterministic != 0, &ws);
    return ws.bytes;
}

namespace gs {
// Shared by the other translation units: bind the workspace for a problem size.
gs_status bind_workspace(void* base, size_t bytes, int64_t n_gauss, int64_t capacity,
                         const gs_grid* grid, const gs_config* cfg, Workspace* ws) {
    if (!base) return GS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(base) % 256 != 0) return GS_ERR_INVALID_ARG;
    carve_workspace(nullptr, n_gauss, capacity, n_bricks_of(grid, cfg), n_voxels_of(grid),
                    cfg->deterministic != 0, ws);
    if (bytes < ws->bytes) return GS_ERR_WORKSPACE;
    carve_workspace(base, n_gauss, capacity, n_bricks_of(grid, cfg), n_voxels_of(grid),
                    cfg->deterministic != 0, ws);
    return GS_OK;
}

bool bins_match(const gs_bins* b, const gs_grid* grid, const gs_config* cfg) {
    if (!b || !b->brick_off || !b->pair_gid || !b->pair_gmj || !b->pair_brick || !b->gm_off || !b->rec ||
        !b->brange || !b->d_npairs || !b->d_status)
        return false;
    BrickGeom g = brick_geom(grid, cfg);
    return b->nbx == g.nbx && b->nby == g.nby && b->nbz == g.nbz &&
           b->n_bricks == g.nbx * g.nby * g.nbz && b->capacity >= 0 &&
           b->capacity <= kMaxCapacity && b->n_gauss >= 0;
}

gs_status bin_bricks_impl(const float* params, const gs_grid* grid, const gs_config* cfg,
                          gs_bins* bins, const Workspace& ws, cudaStream_t st) {
    const int64_t N = bins->n_gauss;
    const int64_t cap = bins->capacity;
    BrickGeom b = brick_geom(grid, cfg);
    GridF G;
    G.n[0] = grid->nx; G.n[1] = grid->ny; G.n[2] = grid->nz;
    for (int k = 0; k < 3; ++k) {
        G.h[k] = grid->h[k];
        G.o[k] = grid->origin[k];
        G.ih[k] = 1.0f / grid->h[k];
        int e;
        G.pow2[k] = frexpf(grid->h[k], &e) == 0.5f && e > -100 && e < 100;
    }
    G.b[0] = b.bx; G.b[1] = b.by; G.b[2] = b.bz;
    G.nb[0] = b.nbx; G.nb[1] = b.nby; G.nb[2] = b.nbz;
    for (int k = 0; k < 3; ++k) G.db[k] = make_fastdiv(static_cast<unsigned>(G.b[k]));

    const int64_t off_bytes = sizeof(int32_t) * (int64_t(bins->n_bricks) + 1);
    if (N == 0) {
        if (cudaMemsetAsync(bins->d_status, 0, sizeof(int32_t), st) != cudaSuccess ||
            cudaMemsetAsync(bins->d_npairs, 0, sizeof(int64_t), st) != cudaSuccess ||
            cudaMemsetAsync(bins->gm_off, 0, sizeof(int32_t), st) != cudaSuccess ||
            cudaMemsetAsync(bins->brick_off, 0, off_bytes, st) != cudaSuccess)
            return GS_ERR_CUDA;
        return GS_OK;
    }
    const int passes = ws.radix_passes;
    const int bits0 = pass_bits(ws.key_bits, passes, 0), nd0 = 1 << bits0;
    const int gt = gauss_tile(N);
    const unsigned gb = static_cast<unsigned>((N + gt - 1) / gt);
    launch_k(gt == 64 ? k_preprocess<64> : k_preprocess<256>, dim3(gb), dim3(gt), 0, st, params, N, G, cfg->trunc_sigma,
        cfg->signal_mode, cfg->a_act, cfg->t_act, bins->rec, bins->brange, nd0, ws.hist0, ws.stride0,
        ws.blk_base);
    gs_status s = last_launch_status();
    if (s != GS_OK) return s;
    const unsigned tiles = static_cast<unsigned>((cap + kSortTile - 1) / kSortTile);
    // Blocks for the parts of heavy tiles (no tile is heavy where its Gaussians on all bricks, or the
    // capacity, are no more than a part). They follow the tiles' blocks, or, where the tiles are more
    // than two per SM but fewer than the resident blocks and may take several rounds, in a launch of
    // their own: more blocks than tiles there put a fourth tile on a few SMs (391 tiles of three rounds
    // 101 -> 110 us; the launch costs 2 us).
    const int64_t max_tile = int64_t(gt) * bins->n_bricks < cap ? int64_t(gt) * bins->n_bricks : cap;
    const int64_t max_parts = max_tile > kFirstMinPart ? (cap + kFirstMinPart - 1) / kFirstMinPart : 0;
    const unsigned parts = static_cast<unsigned>(max_parts < kFirstParts ? max_parts : kFirstParts);
    const bool parts_apart = gb > kScatterWave / 2 && gb < kScatterWave && cap > int64_t(gb) * 2 * kFirstRound;
    for (int pass = 0, shift = 0; pass < passes; ++pass) {
        const int bits = pass_bits(ws.key_bits, passes, pass), nd = 1 << bits;
        const size_t smem = sizeof(int) * (kSortThreads / 32 + 1) * nd;
        const bool first = pass == 0, last = pass == passes - 1;
        const int cur = (pass + 1) & 1;  // later passes alternate: pass 1 reads buffers 0, pass 2 buffers 1
        const int nxt = pass & 1;
        const int bits_next = last ? 0 : pass_bits(ws.key_bits, passes, pass + 1);
        const bool count_next = !last && N < kCountCloud;
        RowScan R = {};
        R.hist = first ? ws.hist0 : ws.hist[cur];
        R.stride = first ? ws.stride0 : ws.stride1;
        R.cols = first ? int64_t(gb) : -1;
        R.rowtot = ws.rowtot;
        R.zero = count_next ? ws.hist[nxt] : nullptr;
        R.zero_rows = 1 << bits_next;
        R.zero_stride = ws.stride1;
        R.blk = ws.blk_base;
        R.ticket = ws.ticket;
        R.nd = nd;
        R.npairs = bins->d_npairs;
        R.capacity = cap;
        R.status = bins->d_status;
        if (!first && tiles > 0 && N >= kCountCloud) {
            launch_k(k_tile_count, dim3((tiles + kCountTiles - 1) / kCountTiles), dim3(kSortThreads), 0, st, ws.keys[cur],
                     bins->d_npairs, cap, shift, nd, ws.hist[cur], ws.stride1);
            s = last_launch_status();
            if (s != GS_OK) return s;
        }
        launch_k(k_row_scan, dim3(nd + (first ? 1 : 0)), dim3(kRowThreads), 0, st, R);
        s = last_launch_status();
        if (s != GS_OK) return s;
        Scatter A = {};
        A.keys_in = first ? nullptr : ws.keys[cur];
        A.vals_in = first ? nullptr : ws.vals[cur];
        A.keys_out = last ? bins->pair_brick : ws.keys[nxt];
        A.vals_out = last ? nullptr : ws.vals[nxt];
        A.out_gmj = bins->pair_gmj;
        A.out_gid = bins->pair_gid;
        A.hist = R.hist;
        A.stride = R.stride;
        A.rowtot = ws.rowtot;
        A.hist_next = R.zero;
        A.stride_next = ws.stride1;
        A.bits_next = bits_next;
        A.shift = shift;
        A.bits = bits;
        A.npairs = bins->d_npairs;
        A.capacity = cap;
        A.brange = bins->brange;
        A.gm_off = bins->gm_off;
        A.blk_base = ws.blk_base;
        A.N = N;
        A.tiles = gb;
        A.nbx = b.nbx;
        A.nby = b.nby;
        A.nb = bins->n_bricks;
        A.brick_off = bins->brick_off;
        void (*kern)(Scatter) = !first    ? (last ? k_radix_scatter<false, true, 256> : k_radix_scatter<false, false, 256>)
                                : gt == 64 ? (last ? k_radix_scatter<true, true, 64> : k_radix_scatter<true, false, 64>)
                                           : (last ? k_radix_scatter<true, true, 256> : k_radix_scatter<true, false, 256>);
        if (first || tiles > 0) {
            launch_k(kern, dim3(first ? gb + (parts_apart ? 0 : parts) : tiles), dim3(kSortThreads), smem, st, A);
            s = last_launch_status();
            if (s != GS_OK) return s;
        }
        if (first && parts_apart && parts > 0) {
            A.block0 = gb;
            launch_k(kern, dim3(parts), dim3(kSortThreads), smem, st, A);
            s = last_launch_status();
            if (s != GS_OK) return s;
        }
        shift += bits;
    }
    if (passes == 1) return GS_OK;  // (brick_off is written by the pass)
    if (cap == 0)
        return cudaMemsetAsync(bins->brick_off, 0, off_bytes, st) == cudaSuccess ? GS_OK : GS_ERR_CUDA;
    // enough threads for four keys each, at most eight blocks per SM
    const int64_t ob = (cap / 4 + 256) / 256;
    launch_k(k_brick_off, dim3(static_cast<unsigned>(ob < kSms * 8 ? ob : kSms * 8)), dim3(256), 0, st,
        bins->pair_brick, bins->d_npairs, cap, bins->n_bricks, bins->brick_off);
    return last_launch_status();
}

}  // namespace gs

extern "C" gs_status gs_bin_bricks(const float* params, const gs_grid* grid, const gs_config* cfg,
                                   gs_bins* bins, void* ws, size_t ws_bytes, gs_stream stream) {
    gs_status s = validate_grid_cfg(grid, cfg);
    if (s != GS_OK) return s;
    if (!bins_match(bins, grid, cfg)) return GS_ERR_INVALID_ARG;
    if (bins->n_gauss > 0 && !params) return GS_ERR_INVALID_ARG;
    if (params && reinterpret_cast<uintptr_t>(params) % 16 != 0) return GS_ERR_INVALID_ARG;
    Workspace w;
    s = bind_workspace(ws, ws_bytes, bins->n_gauss, bins->capacity, grid, cfg, &w);
    if (s != GS_OK) return s;
    return bin_bricks_impl(params, grid, cfg, bins, w, reinterpret_cast<cudaStream_t>(stream));
}

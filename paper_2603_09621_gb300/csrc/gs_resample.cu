// gs_resample.cu -- trilinear resize with half-pixel centres (Sec. 4.1 makes the LR inputs
// by trilinear downsampling), its adjoint as a deterministic gather, and the adjoint fused
// with the adjoint render's per-voxel factors for the fitting step.
//
// Along one axis, destination sample j sits at the source continuous index
// c_j = (n_src / n_dst)(j + 1/2) - 1/2 (raised to 0 where negative) and reads source samples
// i0 = floor(c_j), i1 = min(i0 + 1, n_src - 1) with weights 1 - w, w = c_j - i0. c_j is
// formed with one rounding per FP32 operation (no contraction), so every kernel, and the
// oracle, take the same integer decisions.
#include <cuda_runtime.h>
#include <stdint.h>

#include "gs_common.cuh"

namespace gs {

struct ResAxis {
    float scale;  // n_src / n_dst, FP32 division
    float inv;    // n_dst / n_src (only bounds the adjoint's search range)
    int n_src, n_dst;
};

struct ResGeo {
    ResAxis a[3];  // x, y, z
};

__device__ __forceinline__ void res_map(const ResAxis& A, int j, int& i0, int& i1, float& w) {
    float c = __fsub_rn(__fmul_rn(A.scale, __fadd_rn(float(j), 0.5f)), 0.5f);
    c = fmaxf(c, 0.0f);
    const float f = floorf(c);
    i0 = static_cast<int>(f);
    i1 = min(i0 + 1, A.n_src - 1);
    w = __fsub_rn(c, f);  // exact: 0 <= c - f < 1
}

// Weight with which destination sample j reads source sample i (both corners may coincide
// at the upper edge).
__device__ __forceinline__ float res_weight(const ResAxis& A, int j, int i) {
    int i0, i1;
    float w;
    res_map(A, j, i0, i1, w);
    return (i0 == i ? 1.0f - w : 0.0f) + (i1 == i ? w : 0.0f);
}

// Destination samples that may read source sample i: c_j in [i - 1, i + 1), widened by one.
__device__ __forceinline__ void res_range(const ResAxis& A, int i, int& jlo, int& jhi) {
    jlo = max(0, static_cast<int>(floorf((float(i) - 0.5f) * A.inv - 0.5f)) - 1);
    jhi = min(A.n_dst - 1, static_cast<int>(ceilf((float(i) + 1.5f) * A.inv - 0.5f)) + 1);
}

// Threads along a row of n pieces: up to 256 in whole warps, or the power of two that covers a short row.
__host__ __device__ inline int row_threads(int n) {
    if (n >= 32) return n >= 256 ? 256 : (n + 31) / 32 * 32;
    int t = 1;
    while (t < n) t *= 2;
    return t;
}

// A thread owns one destination column x of a plane z and walks kRows rows y: its x and z taps are
// formed once, and an element offset (T: 32 bits where the source allows) is a sum of precomputed
// parts. Bound by instruction issue: one voxel per thread with three index remainders and 64-bit
// addresses took 170 instructions a voxel. L2 flushed, before -> one row -> four rows per thread:
// 240 x 240 x 155 to 100^3 14.3 -> 13.6 -> 18.4 us (too few warps in flight), to 200 x 200 x 129
// 40.5 -> 31.2 -> 31.3, 100^3 to 240 x 240 x 155 63.8 -> 45.0 -> 34.9.
constexpr int64_t kFwdRowsMin = 5 << 20;  // destination voxels from which a thread walks four rows

template <typename T, int kRows>
__global__ void __launch_bounds__(256) k_resample_fwd(const float* __restrict__ src, ResGeo G,
                                                      float* __restrict__ dst) {
    pdl_enter();
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= AX.n_dst) return;
    int x0, x1;
    float wx;
    res_map(AX, x, x0, x1, wx);
    const float ux = 1.0f - wx;
    const T sx = T(AX.n_src), sxy = sx * T(AY.n_src);
    for (int z = blockIdx.z * blockDim.z + threadIdx.z; z < AZ.n_dst; z += gridDim.z * blockDim.z) {
        int z0, z1;
        float wz;
        res_map(AZ, z, z0, z1, wz);
        const float uz = 1.0f - wz;
        const T a0 = T(z0) * sxy + T(x0), a1 = T(z1) * sxy + T(x0);  // sample x0 of row 0 in each plane
        const T dx = T(x1) - T(x0);
        const int64_t out = int64_t(z) * AY.n_dst * AX.n_dst + x;
        for (int yb = (blockIdx.y * blockDim.y + threadIdx.y) * kRows; yb < AY.n_dst;
             yb += gridDim.y * blockDim.y * kRows) {
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const int y = yb + r;
                if (y >= AY.n_dst) break;
                int y0, y1;
                float wy;
                res_map(AY, y, y0, y1, wy);
                const T b0 = T(y0) * sx, b1 = T(y1) * sx;
                const float uy = 1.0f - wy;
                const float r00 = fmaf(wx, src[a0 + b0 + dx], ux * src[a0 + b0]);
                const float r01 = fmaf(wx, src[a0 + b1 + dx], ux * src[a0 + b1]);
                const float r10 = fmaf(wx, src[a1 + b0 + dx], ux * src[a1 + b0]);
                const float r11 = fmaf(wx, src[a1 + b1 + dx], ux * src[a1 + b1]);
                const float s0 = fmaf(wy, r01, uy * r00);
                const float s1 = fmaf(wy, r11, uy * r10);
                dst[out + int64_t(y) * AX.n_dst] = fmaf(wz, s1, uz * s0);
            }
        }
    }
}

// The destination samples that read source sample i form one run j0, j0 + 1, ... (i0(j) is
// non-decreasing in j). K slots cover it under the bounds of res_list_ok / res_two_taps.
// Slot k holds the weight of j0 + k (0 past the run); *n is the run length.
constexpr int kResList = 4;
template <int K = kResList>
__device__ __forceinline__ void res_list(const ResAxis& A, int i, int& j0, int& n, float (&w)[K]) {
    int lo, hi;
    res_range(A, i, lo, hi);
    int t = lo;
    for (; t < hi; ++t) {  // skip samples whose upper corner is still below i
        int a, b;
        float ww;
        res_map(A, t, a, b, ww);
        if (b >= i) break;
    }
    j0 = t;
    n = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int j = t + k;
        w[k] = (j < A.n_dst) ? res_weight(A, j, i) : 0.0f;
        n = (w[k] != 0.0f) ? k + 1 : n;
    }
}

// Run lengths with FP32 positions: c_j is within c 2^-23 of its exact value, so for source
// sizes up to 2^16 consecutive positions are spaced by the scale +- 2^-6.
//   kResList slots: scale >= 2/3 on every axis keeps the spacing above 0.65, so at most
//   four positions fall in one window [i - 1, i + 1).
//   2 slots: an exact copy (scale 1: c_j = j) or scale >= 1.05 (spacing above 1.03).
constexpr int kResMaxSrc = 1 << 16;
static bool res_list_ok(const ResGeo& G) {
    for (int a = 0; a < 3; ++a)
        if (!(G.a[a].inv <= 1.5f) || G.a[a].n_src > kResMaxSrc) return false;
    return true;
}

static bool res_two_taps(const ResGeo& G) {
    for (int a = 0; a < 3; ++a) {
        const ResAxis& A = G.a[a];
        if (A.n_src > kResMaxSrc) return false;
        if (A.n_dst != A.n_src && !(A.scale >= 1.05f)) return false;
    }
    return true;
}

// Adjoint value at source voxel (x, y, z): sum over the destination samples that read it, in
// ascending (z, y, x) order (any ratio).
__device__ __forceinline__ float res_gather(const float* __restrict__ ddst, const ResGeo& G, int x,
                                            int y, int z) {
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    int xlo, xhi, ylo, yhi, zlo, zhi;
    res_range(AX, x, xlo, xhi);
    res_range(AY, y, ylo, yhi);
    res_range(AZ, z, zlo, zhi);
    float acc = 0.0f;
    for (int jz = zlo; jz <= zhi; ++jz) {
        const float wz = res_weight(AZ, jz, z);
        if (wz == 0.0f) continue;
        for (int jy = ylo; jy <= yhi; ++jy) {
            const float wy = res_weight(AY, jy, y);
            if (wy == 0.0f) continue;
            const float wzy = wz * wy;
            const float* row = ddst + (int64_t(jz) * AY.n_dst + jy) * AX.n_dst;
            for (int jx = xlo; jx <= xhi; ++jx) {
                const float wx = res_weight(AX, jx, x);
                if (wx != 0.0f) acc = fmaf(wzy * wx, row[jx], acc);
            }
        }
    }
    return acc;
}

__global__ void __launch_bounds__(256) k_resample_bwd(const float* __restrict__ ddst, ResGeo G,
                                                      float* __restrict__ dsrc) {
    pdl_enter();
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    const int64_t n = int64_t(AX.n_src) * AY.n_src * AZ.n_src;
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n;
         t += int64_t(gridDim.x) * blockDim.x) {
        const int x = static_cast<int>(t % AX.n_src);
        const int y = static_cast<int>((t / AX.n_src) % AY.n_src);
        const int z = static_cast<int>(t / (int64_t(AX.n_src) * AY.n_src));
        dsrc[t] = res_gather(ddst, G, x, y, z);
    }
}

// Table form of the adjoint gather (under res_list_ok / res_two_taps, with at most
// kResTabMax source samples over the three axes): each block tabulates the runs of every
// source x, y and z in shared memory once, then sweeps source rows (z, y) with one thread
// per voxel; a voxel reads its three runs from the tables and gathers in ascending (z, y, x)
// order.
constexpr int kResTabMax = 2048;

template <int K>
struct ResRun {
    int j0, n;
    float w[K];
};

template <bool kPrep, int K>
__global__ void __launch_bounds__(256) k_resample_adj_tab(const float* __restrict__ ddst, ResGeo G,
                                                          const float* __restrict__ Iv,
                                                          const float* __restrict__ Wv, float eps,
                                                          float* __restrict__ dsrc,
                                                          float2* __restrict__ aip) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char res_smem[];
    ResRun<K>* tab = reinterpret_cast<ResRun<K>*>(res_smem);
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    const int nx = AX.n_src, ny = AY.n_src, nz = AZ.n_src;
    ResRun<K>* xt = tab;
    ResRun<K>* yt = tab + nx;
    ResRun<K>* zt = tab + nx + ny;
    for (int e = threadIdx.x; e < nx + ny + nz; e += blockDim.x) {
        const int ax = e < nx ? 0 : (e < nx + ny ? 1 : 2);
        const int i = e - (ax > 0 ? nx : 0) - (ax > 1 ? ny : 0);
        ResAxis A;
        A.scale = ax == 0 ? AX.scale : (ax == 1 ? AY.scale : AZ.scale);
        A.inv = ax == 0 ? AX.inv : (ax == 1 ? AY.inv : AZ.inv);
        A.n_src = ax == 0 ? AX.n_src : (ax == 1 ? AY.n_src : AZ.n_src);
        A.n_dst = ax == 0 ? AX.n_dst : (ax == 1 ? AY.n_dst : AZ.n_dst);
        ResRun<K> rr;
        res_list<K>(A, i, rr.j0, rr.n, rr.w);
        tab[e] = rr;
    }
    __syncthreads();
    const int64_t rows = int64_t(nz) * ny;
    for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
        const int z = static_cast<int>(row / ny), y = static_cast<int>(row - int64_t(z) * ny);
        const ResRun<K> rz = zt[z], ry = yt[y];
        const int64_t row0 = row * nx;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) {
            const ResRun<K> rx = xt[x];
            float acc = 0.0f;
#pragma unroll
            for (int a = 0; a < K; ++a) {
                if (a >= rz.n) break;
#pragma unroll
                for (int b = 0; b < K; ++b) {
                    if (b >= ry.n) break;
                    const float wzy = rz.w[a] * ry.w[b];
                    const float* src =
                        ddst + (int64_t(rz.j0 + a) * AY.n_dst + (ry.j0 + b)) * AX.n_dst + rx.j0;
#pragma unroll
                    for (int c = 0; c < K; ++c) {
                        if (c >= rx.n) break;
                        if (rx.w[c] != 0.0f) acc = fmaf(wzy * rx.w[c], src[c], acc);
                    }
                }
            }
            if (kPrep) {
                const float w = Wv[row0 + x];
                const float al = acc / (w > eps ? w : eps);
                aip[row0 + x] = make_float2(al, (w > eps) ? al * Iv[row0 + x] : 0.0f);
            } else {
                dsrc[row0 + x] = acc;
            }
        }
    }
}

// Fitting step, any ratio: dL/dI at each HR voxel is the resize adjoint of dL/dLR; stored
// directly as the adjoint render's factors (alpha, alpha I'), alpha = dL/dI / max(W, eps),
// I' = I where W > eps, else 0.
__global__ void __launch_bounds__(256) k_resample_adj_prep(const float* __restrict__ dlr, ResGeo G,
                                                           const float* __restrict__ Iv,
                                                           const float* __restrict__ Wv, float eps,
                                                           float2* __restrict__ aip) {
    pdl_enter();
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    const int64_t n = int64_t(AX.n_src) * AY.n_src * AZ.n_src;
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n;
         t += int64_t(gridDim.x) * blockDim.x) {
        const int x = static_cast<int>(t % AX.n_src);
        const int y = static_cast<int>((t / AX.n_src) % AY.n_src);
        const int z = static_cast<int>(t / (int64_t(AX.n_src) * AY.n_src));
        const float gI = res_gather(dlr, G, x, y, z);
        const float w = Wv[t];
        const float al = gI / (w > eps ? w : eps);
        aip[t] = make_float2(al, (w > eps) ? al * Iv[t] : 0.0f);
    }
}

static bool dims_ok(int32_t nz, int32_t ny, int32_t nx) {
    return nz > 0 && ny > 0 && nx > 0 && nx < (1 << 23) && ny < (1 << 23) && nz < (1 << 23);
}

static ResGeo make_res(int32_t snz, int32_t sny, int32_t snx, int32_t dnz, int32_t dny, int32_t dnx) {
    ResGeo G;
    const int32_t s[3] = {snx, sny, snz}, d[3] = {dnx, dny, dnz};
    for (int a = 0; a < 3; ++a) {
        G.a[a].n_src = s[a];
        G.a[a].n_dst = d[a];
        G.a[a].scale = float(s[a]) / float(d[a]);
        G.a[a].inv = float(d[a]) / float(s[a]);
    }
    return G;
}

static unsigned res_blocks(int64_t n) {
    const int64_t b = (n + 255) / 256;
    return static_cast<unsigned>(b < kSms * 64 ? b : kSms * 64);
}

gs_status resample_fwd_impl(const float* src, int32_t snz, int32_t sny, int32_t snx, float* dst,
                            int32_t dnz, int32_t dny, int32_t dnx, cudaStream_t st) {
    const ResGeo G = make_res(snz, sny, snx, dnz, dny, dnx);
    const bool narrow = int64_t(snz) * sny * snx <= (int64_t(1) << 31) - 1;
    const bool rows4 = int64_t(dnz) * dny * dnx >= kFwdRowsMin;
    // a block's threads over columns (whole warps, or a power of two of a narrow volume's), then rows,
    // then planes: with whole warps along any row 1,024 x 1,024 samples of one column took 146 us, 15 now
    const int tx = row_threads(dnx), rows = rows4 ? 4 : 1;
    int ty = 1, tz = 1;
    while (2 * ty * tx <= 256 && ty * rows < dny) ty *= 2;
    while (2 * tz * ty * tx <= 256 && tz < dnz && tz < 64) tz *= 2;
    const int64_t gx = (int64_t(dnx) + tx - 1) / tx, gy = (int64_t(dny) + ty * rows - 1) / (ty * rows);
    const int64_t gz = (int64_t(dnz) + tz - 1) / tz;
    const dim3 grid(static_cast<unsigned>(gx), static_cast<unsigned>(gy < 65535 ? gy : 65535),
                    static_cast<unsigned>(gz < 65535 ? gz : 65535));
    launch_k(narrow ? (rows4 ? k_resample_fwd<unsigned, 4> : k_resample_fwd<unsigned, 1>)
                    : (rows4 ? k_resample_fwd<int64_t, 4> : k_resample_fwd<int64_t, 1>),
        grid, dim3(tx, ty, tz), 0, st, src, G, dst);
    return last_launch_status();
}

// Separable form of the adjoint for a tile of kRows source rows on each of up to kPlanes source planes z,
// in shared memory: V[j][jx] = sum over the z run of w_z dL/dLR[jz][jy][jx] for the LR rows jy that the
// tile's rows read (each LR value is loaded once per tile), U[y][jx] = sum over the y run of w_y V, then
// each voxel sums its x run over U[y]. Fixed order: z, then y, then x. A thread owns kV consecutive x of
// every (256 / threads per row)-th row: its x runs stay in registers, and with kV = 4 (rows of whole,
// aligned quads) I, W and the factors move by 16-byte accesses. Bound by HBM where it forms the adjoint
// render's factors (143 MB at 240 x 240 x 155 from 100^3: 21 us at the copy bandwidth).
// With z and y taps gathered per (y, jx) from global memory, one voxel per thread, an index division per
// voxel and 1,240 blocks for 1,216 resident ones it took 62 us (26 us without the factors); 36 (16) us
// now. Tiles of 16 (24, 48) rows took 41 (43, 44) us; one plane per block, which forms the x runs twice
// as often, 38 us; kept where two would leave SMs idle.
constexpr int kPlanes = 2;

template <bool kPrep, int K, int kRows, int kV>
__global__ void __launch_bounds__(256) k_resample_adj_plane(const float* __restrict__ ddst, ResGeo G,
                                                            int v_rows, int per, const float* __restrict__ Iv,
                                                            const float* __restrict__ Wv, float eps,
                                                            float* __restrict__ dsrc,
                                                            float2* __restrict__ aip) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char res_smem[];
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    const int nx = AX.n_src, ny = AY.n_src;
    const int lnx = AX.n_dst, lny = AY.n_dst;
    ResRun<K>* xt = reinterpret_cast<ResRun<K>*>(res_smem);
    ResRun<K>* yt = xt + nx;                           // kRows entries
    float* U = reinterpret_cast<float*>(yt + kRows);  // [kRows][lnx]
    float* V = U + kRows * lnx;                       // [v_rows][lnx]
    __shared__ ResRun<K> zt[kPlanes];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int y0 = blockIdx.y * kRows;
    const int rows = min(kRows, ny - y0);
    const int zb = blockIdx.x * per, planes = min(per, AZ.n_src - zb);  // per <= kPlanes
    for (int e = tid; e < nx + rows + planes; e += 256) {
        ResRun<K> rr;
        if (e < nx) {
            res_list<K>(AX, e, rr.j0, rr.n, rr.w);
            xt[e] = rr;
        } else if (e < nx + rows) {
            res_list<K>(AY, y0 + (e - nx), rr.j0, rr.n, rr.w);
            yt[e - nx] = rr;
        } else {
            res_list<K>(AZ, zb + (e - nx - rows), rr.j0, rr.n, rr.w);
            zt[e - nx - rows] = rr;
        }
    }
    __syncthreads();
    const int groups = (nx + kV - 1) / kV;  // kV divides nx where kV > 1
    const int per_row = groups >= 256 ? 256 : (groups + 31) / 32 * 32;
    const int step = 256 / per_row, ty = tid / per_row;
    for (int z = zb; z < zb + planes; ++z) {
        const ResRun<K> zr = zt[z - zb];
        if (zr.n == 0) {
            // no LR sample reads the plane (two in three where z is resized by 3): zero over one run of
            // voxels
            const float none[kV] = {};
            for (int e = tid; e < rows * groups; e += 256)
                emit_voxels<kPrep, kV>((int64_t(z) * ny + y0) * nx + int64_t(e) * kV, none, Iv, Wv, eps, dsrc, aip);
            continue;
        }
        // LR rows of the tile: runs start in ascending order, so rows jf .. jf + nv - 1 (v_rows bounds them)
        const int jf = min(yt[0].j0, lny - 1);
        const int nv = min(min(yt[rows - 1].j0 + K, lny) - jf, v_rows);
        for (int r = warp; r < nv; r += 8)
            for (int jx = lane; jx < lnx; jx += 32) {
                float acc = 0.0f;
#pragma unroll
                for (int a = 0; a < K; ++a)
                    if (a < zr.n) acc = fmaf(zr.w[a], ddst[(int64_t(zr.j0 + a) * lny + jf + r) * lnx + jx], acc);
                V[r * lnx + jx] = acc;
            }
        __syncthreads();
        for (int r = warp; r < rows; r += 8) {
            const ResRun<K> ry = yt[r];
            for (int jx = lane; jx < lnx; jx += 32) {
                float acc = 0.0f;
#pragma unroll
                for (int b = 0; b < K; ++b)
                    if (b < ry.n) acc = fmaf(ry.w[b], V[min(ry.j0 + b - jf, v_rows - 1) * lnx + jx], acc);
                U[r * lnx + jx] = acc;
            }
        }
        __syncthreads();
        for (int gx = tid - ty * per_row; ty < step && gx < groups; gx += per_row) {
            ResRun<K> rx[kV];
#pragma unroll
            for (int e = 0; e < kV; ++e) rx[e] = xt[gx * kV + e];
#pragma unroll 2
            for (int r = ty; r < rows; r += step) {
                const float* u = U + r * lnx;
                float acc[kV];
#pragma unroll
                for (int e = 0; e < kV; ++e) {
                    acc[e] = 0.0f;
#pragma unroll
                    for (int c = 0; c < K; ++c)
                        if (c < rx[e].n) acc[e] = fmaf(rx[e].w[c], u[rx[e].j0 + c], acc[e]);
                }
                const int64_t v = (int64_t(z) * ny + (y0 + r)) * nx + gx * kV;
                emit_voxels<kPrep, kV>(v, acc, Iv, Wv, eps, dsrc, aip);
            }
        }
    }
}

// The same sums for narrow volumes, of up to kThinRow columns. Their tiles are small, and the latency of
// the phases and the lanes without a sample count: U is formed from the LR values in memory, without V
// and its barrier, and the threads run over a tile's samples and voxels without regard to rows. 512 x 300
// planes of 20 columns, from as many (from a third of the planes): 37 (37) us by the plane kernel, 27
// (17) here; of 48 columns 49 (46) and 52 (27), of 60 45 (25 with the empty planes left out) and 58 (31).
// Tiles of 128 rows up to 20 columns, else of 32 (one column of 2,048 x 2,048 from 1,024 x 1,024: 186 us
// with 32, 60 here).
constexpr int kThinRow = 56;
constexpr int kThinTile = 128;

template <bool kPrep, int K, int kV>
__global__ void __launch_bounds__(256) k_resample_adj_thin(const float* __restrict__ ddst, ResGeo G, int tile,
                                                           int per, FastDiv by_lnx, FastDiv by_groups,
                                                           const float* __restrict__ Iv,
                                                           const float* __restrict__ Wv, float eps,
                                                           float* __restrict__ dsrc, float2* __restrict__ aip) {
    pdl_enter();
    const ResAxis &AX = G.a[0], &AY = G.a[1], &AZ = G.a[2];
    const int nx = AX.n_src, ny = AY.n_src, lnx = AX.n_dst, lny = AY.n_dst;
    __shared__ ResRun<K> xt[kThinRow], yt[kThinTile], zt[kPlanes];
    extern __shared__ __align__(16) unsigned char res_smem[];
    float* U = reinterpret_cast<float*>(res_smem);  // [rows][lnx]
    const int tid = threadIdx.x;
    const int y0 = blockIdx.y * tile, rows = min(tile, ny - y0);  // tile <= kThinTile
    const int zb = blockIdx.x * per, planes = min(per, AZ.n_src - zb);  // per <= kPlanes
    for (int e = tid; e < nx + rows + planes; e += 256) {
        ResRun<K> rr;
        if (e < nx) {
            res_list<K>(AX, e, rr.j0, rr.n, rr.w);
            xt[e] = rr;
        } else if (e < nx + rows) {
            res_list<K>(AY, y0 + (e - nx), rr.j0, rr.n, rr.w);
            yt[e - nx] = rr;
        } else {
            res_list<K>(AZ, zb + (e - nx - rows), rr.j0, rr.n, rr.w);
            zt[e - nx - rows] = rr;
        }
    }
    __syncthreads();
    const int groups = nx / kV;  // kV divides nx
    for (int z = zb; z < zb + planes; ++z) {
        const ResRun<K> zr = zt[z - zb];
        const int64_t v0 = (int64_t(z) * ny + y0) * nx;
        if (zr.n == 0) {
            const float none[kV] = {};
            for (int e = tid; e < rows * groups; e += 256)
                emit_voxels<kPrep, kV>(v0 + int64_t(e) * kV, none, Iv, Wv, eps, dsrc, aip);
            continue;
        }
        if (z > zb) __syncthreads();  // U is no longer read
        for (int e = tid; e < rows * lnx; e += 256) {
            const int r = static_cast<int>(fast_div(static_cast<unsigned>(e), by_lnx)), jx = e - r * lnx;
            const ResRun<K> ry = yt[r];
            float acc = 0.0f;
#pragma unroll
            for (int b = 0; b < K; ++b) {
                if (b >= ry.n) break;
                float v = 0.0f;
#pragma unroll
                for (int a = 0; a < K; ++a)
                    if (a < zr.n) v = fmaf(zr.w[a], ddst[(int64_t(zr.j0 + a) * lny + ry.j0 + b) * lnx + jx], v);
                acc = fmaf(ry.w[b], v, acc);
            }
            U[e] = acc;
        }
        __syncthreads();
        for (int e = tid; e < rows * groups; e += 256) {
            const int r = static_cast<int>(fast_div(static_cast<unsigned>(e), by_groups)), gx = e - r * groups;
            const float* u = U + r * lnx;
            float acc[kV];
#pragma unroll
            for (int k = 0; k < kV; ++k) {
                const ResRun<K> rx = xt[gx * kV + k];
                acc[k] = 0.0f;
#pragma unroll
                for (int c = 0; c < K; ++c)
                    if (c < rx.n) acc[k] = fmaf(rx.w[c], u[rx.j0 + c], acc[k]);
            }
            emit_voxels<kPrep, kV>(v0 + int64_t(e) * kV, acc, Iv, Wv, eps, dsrc, aip);
        }
    }
}

// Shared memory of a tile (the kernel also holds the z run): 32 rows as long as five blocks fit an SM,
// else 8 rows as long as two do, which takes volumes of up to about 1,000 columns (512 x 512 x 256 from
// 512 x 512 x 64, 54 KB: 271 us by the run tables, 128 by the plane kernel).
constexpr int kPlaneSmem = 48 * 1024 - 512;
constexpr int kPlaneSmemMax = 112 * 1024;

static int planes_per_block(int64_t nz, int64_t tiles) { return nz * tiles >= kSms * 6 ? kPlanes : 1; }

template <bool kPrep>
static bool vec_volume(const ResGeo& G, const float* I, const float* W, const float* dsrc, const float2* aip) {
    return G.a[0].n_src % 4 == 0 && (kPrep ? aligned16(I) && aligned16(W) && aligned16(aip) : aligned16(dsrc));
}

// Rows per tile: the more, the fewer LR values are read again, but the fewer blocks there are and the
// more shared memory each takes.
template <bool kPrep, int K, int kRows>
static bool launch_adj_plane_rows(const float* dd, const ResGeo& G, const float* I, const float* W, float eps,
                                  float* dsrc, float2* aip, cudaStream_t st) {
    const int nx = G.a[0].n_src, ny = G.a[1].n_src, nz = G.a[2].n_src, lnx = G.a[0].n_dst;
    // LR rows that a tile's rows read: first samples of consecutive rows are n_dst / n_src apart on
    // average, each within two samples of its exact position
    const int v_rows = static_cast<int>((kRows - 1) * G.a[1].inv) + 5 + K;
    const size_t smem = sizeof(ResRun<K>) * (size_t(nx) + kRows) + sizeof(float) * lnx * (size_t(kRows) + v_rows);
    const int64_t tiles = (ny + kRows - 1) / kRows;
    if (smem > size_t(kRows > 8 ? kPlaneSmem : kPlaneSmemMax) || tiles > 65535) return false;
    const int per = planes_per_block(nz, tiles);
    const auto kernel = vec_volume<kPrep>(G, I, W, dsrc, aip) ? k_resample_adj_plane<kPrep, K, kRows, 4>
                                                             : k_resample_adj_plane<kPrep, K, kRows, 1>;
    // (an attribute of the kernel on the current device; beyond 48 KB only)
    if (smem > size_t(kPlaneSmem) &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
        return false;
    launch_k(kernel, dim3(static_cast<unsigned>((nz + per - 1) / per), static_cast<unsigned>(tiles)), dim3(256), smem,
        st, dd, G, v_rows, per, I, W, eps, dsrc, aip);
    return true;
}

template <bool kPrep, int K>
static bool launch_adj_thin(const float* dd, const ResGeo& G, const float* I, const float* W, float eps, float* dsrc,
                            float2* aip, cudaStream_t st) {
    const int nx = G.a[0].n_src, ny = G.a[1].n_src, nz = G.a[2].n_src, lnx = G.a[0].n_dst;
    const int tile = nx <= 20 ? kThinTile : 32;
    const int64_t tiles = (ny + tile - 1) / tile;
    if (nx > kThinRow || tiles > 65535) return false;
    const int per = planes_per_block(nz, tiles);
    const bool vec = vec_volume<kPrep>(G, I, W, dsrc, aip);
    launch_k(vec ? k_resample_adj_thin<kPrep, K, 4> : k_resample_adj_thin<kPrep, K, 1>,
        dim3(static_cast<unsigned>((nz + per - 1) / per), static_cast<unsigned>(tiles)), dim3(256),
        sizeof(float) * tile * lnx, st, dd, G, tile, per, make_fastdiv(static_cast<unsigned>(lnx)),
        make_fastdiv(static_cast<unsigned>(vec ? nx / 4 : nx)), I, W, eps, dsrc, aip);
    return true;
}

template <bool kPrep, int K>
static bool launch_adj_plane_k(const float* dd, const ResGeo& G, const float* I, const float* W,
                               float eps, float* dsrc, float2* aip, cudaStream_t st) {
    return launch_adj_thin<kPrep, K>(dd, G, I, W, eps, dsrc, aip, st) ||
           launch_adj_plane_rows<kPrep, K, 32>(dd, G, I, W, eps, dsrc, aip, st) ||
           launch_adj_plane_rows<kPrep, K, 8>(dd, G, I, W, eps, dsrc, aip, st);
}

template <bool kPrep>
static bool launch_adj_plane(const float* dd, const ResGeo& G, const float* I, const float* W,
                             float eps, float* dsrc, float2* aip, cudaStream_t st) {
    if (!res_list_ok(G)) return false;
    if (res_two_taps(G)) return launch_adj_plane_k<kPrep, 2>(dd, G, I, W, eps, dsrc, aip, st);
    return launch_adj_plane_k<kPrep, kResList>(dd, G, I, W, eps, dsrc, aip, st);
}

template <bool kPrep>
static bool launch_adj_tab(const float* dd, const ResGeo& G, const float* I, const float* W,
                           float eps, float* dsrc, float2* aip, cudaStream_t st) {
    const int n_tab = G.a[0].n_src + G.a[1].n_src + G.a[2].n_src;
    if (!res_list_ok(G) || n_tab > kResTabMax) return false;
    const int64_t rows = int64_t(G.a[2].n_src) * G.a[1].n_src;
    const unsigned nb = static_cast<unsigned>(rows < kSms * 8 ? rows : kSms * 8);
    if (res_two_taps(G))
        launch_k(k_resample_adj_tab<kPrep, 2>, dim3(nb), dim3(256), sizeof(ResRun<2>) * n_tab, st,
            dd, G, I, W, eps, dsrc, aip);
    else
        launch_k(k_resample_adj_tab<kPrep, kResList>, dim3(nb), dim3(256),
            sizeof(ResRun<kResList>) * n_tab, st, dd, G, I, W, eps, dsrc, aip);
    return true;
}

gs_status resample_adj_prep_impl(const float* dlr, int32_t lnz, int32_t lny, int32_t lnx,
                                 const float* I, const float* W, int32_t nz, int32_t ny, int32_t nx,
                                 float eps, float2* aip, cudaStream_t st) {
    const ResGeo G = make_res(nz, ny, nx, lnz, lny, lnx);
    if (!launch_adj_plane<true>(dlr, G, I, W, eps, nullptr, aip, st) &&
        !launch_adj_tab<true>(dlr, G, I, W, eps, nullptr, aip, st))
        launch_k(k_resample_adj_prep, dim3(res_blocks(int64_t(nz) * ny * nx)), dim3(256), 0, st,
            dlr, G, I, W, eps, aip);
    return last_launch_status();
}

}  // namespace gs

using namespace gs;

extern "C" gs_status gs_resample_fwd(const float* src, int32_t snz, int32_t sny, int32_t snx,
                                     float* dst, int32_t dnz, int32_t dny, int32_t dnx,
                                     gs_stream stream) {
    if (!src || !dst || !dims_ok(snz, sny, snx) || !dims_ok(dnz, dny, dnx)) return GS_ERR_INVALID_ARG;
    return resample_fwd_impl(src, snz, sny, snx, dst, dnz, dny, dnx,
                             reinterpret_cast<cudaStream_t>(stream));
}

extern "C" gs_status gs_resample_bwd(const float* ddst, int32_t dnz, int32_t dny, int32_t dnx,
                                     float* dsrc, int32_t snz, int32_t sny, int32_t snx,
                                     gs_stream stream) {
    if (!ddst || !dsrc || !dims_ok(snz, sny, snx) || !dims_ok(dnz, dny, dnx)) return GS_ERR_INVALID_ARG;
    const ResGeo G = make_res(snz, sny, snx, dnz, dny, dnx);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (!launch_adj_plane<false>(ddst, G, nullptr, nullptr, 0.f, dsrc, nullptr, st) &&
        !launch_adj_tab<false>(ddst, G, nullptr, nullptr, 0.f, dsrc, nullptr, st))
        launch_k(k_resample_bwd, dim3(res_blocks(int64_t(snz) * sny * snx)), dim3(256), 0, st, ddst,
            G, dsrc);
    return last_launch_status();
}

// gs_volume.cu -- slice-profile forward model (box average of s slices along z), its
// adjoint, the deterministic L1 loss, the fused fitting step and the small host utilities of
// the C ABI.
#include <cuda_runtime.h>

#include <mutex>
#include <stdint.h>

#include <atomic>

#include "gs_common.cuh"

namespace gs {

static std::atomic<unsigned long long> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

// Slice profile and its adjoint over a 2D grid of 2D blocks: y strides over the LR slices, a thread
// owns kV consecutive voxels of a plane (4: 16-byte accesses, for aligned volumes whose planes
// are a multiple of 4 voxels; else 1), so no voxel needs an index division. Bound by HBM. The
// adjoint reads each LR value once for its s HR slices and took 33 us with one HR voxel and two
// 64-bit divisions per thread at 192 x 192 x 128, s = 2; 5 us now (28 MB).
template <int kV>
struct Voxels {
    float v[kV];
};

template <int kV>
__device__ __forceinline__ Voxels<kV> load_voxels(const float* src) {
    Voxels<kV> r;
    if constexpr (kV == 4)
        load4<true>(src, r.v);
    else
        r.v[0] = *src;
    return r;
}

template <int kV>
__device__ __forceinline__ void store_voxels(float* dst, const Voxels<kV>& r) {
    if constexpr (kV == 4)
        store4<true>(dst, r.v);
    else
        *dst = r.v[0];
}

// kS: slices per LR slice at compile time, their loads in flight together (0: any number s_, four or six at a
// time). With the loop left to the compiler two slices took 23 us where 18 are enough (300 x 256 x 256).
template <int kV, int kS>
__global__ void __launch_bounds__(256) k_downsample_fwd(const float* __restrict__ hr, unsigned plane,
                                                        unsigned nzl, int s_, float inv_s,
                                                        float* __restrict__ lr) {
    pdl_enter();
    constexpr int kBatch = kS > 0 ? kS : (kV == 4 ? 4 : 6);
    const int s = kS > 0 ? kS : s_;
    for (unsigned k = blockIdx.y * blockDim.y + threadIdx.y; k < nzl; k += gridDim.y * blockDim.y) {
        const float* src = hr + int64_t(k) * s * plane;
        for (unsigned r = (blockIdx.x * blockDim.x + threadIdx.x) * kV; r < plane; r += gridDim.x * blockDim.x * kV) {
            Voxels<kV> acc = {};
            for (int j0 = 0; j0 < s; j0 += kBatch) {
                Voxels<kV> x[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j)
                    if (kS > 0 || j0 + j < s) x[j] = load_voxels<kV>(src + int64_t(j0 + j) * plane + r);
#pragma unroll
                for (int j = 0; j < kBatch; ++j)
                    if (kS > 0 || j0 + j < s)
#pragma unroll
                        for (int e = 0; e < kV; ++e) acc.v[e] += x[j].v[e];
            }
#pragma unroll
            for (int e = 0; e < kV; ++e) acc.v[e] *= inv_s;
            store_voxels<kV>(lr + int64_t(k) * plane + r, acc);
        }
    }
}

// (slice nzl stands for the trailing HR slices, whose gradient is zero)
template <int kV>
__global__ void __launch_bounds__(256) k_downsample_bwd(const float* __restrict__ dlr, int nz, unsigned plane,
                                                        unsigned nzl, int s, float inv_s,
                                                        float* __restrict__ dhr) {
    pdl_enter();
    for (unsigned k = blockIdx.y * blockDim.y + threadIdx.y; k <= nzl; k += gridDim.y * blockDim.y) {
        const int j1 = k < nzl ? s : nz - static_cast<int>(nzl) * s;
        float* dst = dhr + int64_t(k) * s * plane;
        for (unsigned r = (blockIdx.x * blockDim.x + threadIdx.x) * kV; r < plane; r += gridDim.x * blockDim.x * kV) {
            Voxels<kV> x = {};
            if (k < nzl) {
                x = load_voxels<kV>(dlr + int64_t(k) * plane + r);
#pragma unroll
                for (int e = 0; e < kV; ++e) x.v[e] *= inv_s;
            }
            for (int j = 0; j < j1; ++j) store_voxels<kV>(dst + int64_t(j) * plane + r, x);
        }
    }
}

// The adjoint render's factors with the profile's adjoint, one HR slice after the other (the LR values
// are cached).
template <int kV>
__global__ void __launch_bounds__(256) k_profile_factors(const float* __restrict__ dlr, unsigned nz, unsigned plane,
                                                         unsigned nzl, unsigned s, float inv_s,
                                                         const float* __restrict__ Iv,
                                                         const float* __restrict__ Wv, float eps,
                                                         float2* __restrict__ aip) {
    pdl_enter();
    for (unsigned z = blockIdx.y * blockDim.y + threadIdx.y; z < nz; z += gridDim.y * blockDim.y) {
        const unsigned k = z / s;
        for (unsigned r = (blockIdx.x * blockDim.x + threadIdx.x) * kV; r < plane; r += gridDim.x * blockDim.x * kV) {
            Voxels<kV> x = {};
            if (k < nzl) {
                x = load_voxels<kV>(dlr + int64_t(k) * plane + r);
#pragma unroll
                for (int e = 0; e < kV; ++e) x.v[e] *= inv_s;
            }
            emit_voxels<true, kV>(int64_t(z) * plane + r, x.v, Iv, Wv, eps, nullptr, aip);
        }
    }
}

// L1 sums: a fixed grid of kL1Blocks blocks of kL1Threads; thread t sums |pred - target| over the
// quads of consecutive values t, t + 131,072, ..., then a fixed-shape tree over the block (partials)
// and over the blocks, so the loss does not depend on which kernel forms it or on alignment. The
// last tree runs in a launch of its own (k_l1_final) or in the block that finishes last (ticket: a
// counter cleared earlier on the stream).
constexpr int kL1Threads = 128;

__device__ __forceinline__ float l1_block_sum(float acc, float* sm) {
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int o = kL1Threads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
        __syncthreads();
    }
    return sm[0];
}

// Tree over the kL1Blocks partials by one block of kL1Threads.
__device__ __forceinline__ void l1_total(const float* partials, float inv_n, float* loss, float* sm) {
    constexpr int kPer = kL1Blocks / kL1Threads;  // partials per thread: the tree's first levels
    const int t = threadIdx.x;
    float p[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) p[k] = __ldcg(partials + t + k * kL1Threads);
#pragma unroll
    for (int o = kPer / 2; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < o; ++k) p[k] += p[k + o];
    const float sum = l1_block_sum(p[0], sm);
    if (t == 0) *loss = sum * inv_n;
}

__device__ __forceinline__ void l1_finish(float acc, float inv_n, float* partials, int* ticket, float* loss) {
    __shared__ float sm[kL1Threads];
    __shared__ bool last;
    const float sum = l1_block_sum(acc, sm);
    if (threadIdx.x == 0) partials[blockIdx.x] = sum;
    if (!ticket) return;
    if (threadIdx.x == 0) {
        __threadfence();  // the partial is visible before the ticket is taken
        last = atomicAdd(ticket, 1) == kL1Blocks - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    l1_total(partials, inv_n, loss, sm);
}

__device__ __forceinline__ float l1_sign(float d, float inv_n) {
    return (d > 0.f) ? inv_n : ((d < 0.f) ? -inv_n : 0.f);
}

// The fitting step's counter: one thread of the loss kernel counts the step (d_step, or nullptr),
// unless the binning overflowed the capacity and the step will change nothing.
struct StepCount {
    int32_t* d_step;
    const int64_t* npairs;
    int64_t capacity;
};

__device__ __forceinline__ void count_step(const StepCount& c) {
    if (c.d_step && blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t P = *c.npairs;
        if (P >= 0 && P <= c.capacity) *c.d_step += 1;
    }
}

// Optionally writes sign(pred - target) / n. kVec: 16-byte accesses of aligned arrays. Bound by HBM: two
// quads of a thread are in flight together, added in their order (67M values with the gradient: 118 us;
// one quad at a time 136, four 125, twice the threads with 4-byte accesses 123).
constexpr int kL1Ahead = 2;

template <bool kVec>
__global__ void __launch_bounds__(kL1Threads) k_l1_partial(const float* __restrict__ pred,
                                                           const float* __restrict__ target, int64_t n,
                                                           float inv_n, float* dpred, float* partials,
                                                           int* ticket, float* loss, StepCount count) {
    pdl_enter();
    count_step(count);
    constexpr int64_t kStep = 4 * kL1Blocks * kL1Threads;
    float acc = 0.f;
    for (int64_t i0 = 4 * (int64_t(blockIdx.x) * kL1Threads + threadIdx.x); i0 < n; i0 += kL1Ahead * kStep) {
        float p[kL1Ahead][4], t[kL1Ahead][4];
#pragma unroll
        for (int u = 0; u < kL1Ahead; ++u)
            if (i0 + u * kStep + 3 < n) {
                load4<kVec>(pred + i0 + u * kStep, p[u]);
                load4<kVec>(target + i0 + u * kStep, t[u]);
            }
#pragma unroll
        for (int u = 0; u < kL1Ahead; ++u) {
            const int64_t i = i0 + u * kStep;
            if (i + 3 < n) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float d = p[u][e] - t[u][e];
                    acc += fabsf(d);
                    p[u][e] = l1_sign(d, inv_n);
                }
                if (dpred) store4<kVec>(dpred + i, p[u]);
            } else {
                for (int64_t e = i; e < n; ++e) {
                    const float d = pred[e] - target[e];
                    acc += fabsf(d);
                    if (dpred) dpred[e] = l1_sign(d, inv_n);
                }
            }
        }
    }
    l1_finish(acc, inv_n, partials, ticket, loss);
}

__global__ void __launch_bounds__(kL1Threads) k_l1_final(const float* partials, float inv_n, float* loss) {
    pdl_enter();
    __shared__ float sm[kL1Threads];
    l1_total(partials, inv_n, loss, sm);
}

// The fitting step's z box model in one pass: slice profile, L1 and its sign gradient (to lr_pred),
// profile adjoint and the adjoint render's factors (alpha, alpha I') of the s HR voxels below each LR
// voxel, with dL/dI = dL/dLR / s (0 in the trailing slices, which no LR slice covers). Bound by HBM: I,
// W, target read once, dL/dLR and the factors written once. kS: slices per LR slice, whose I values stay
// in registers. A thread owns a quad of LR voxels as in k_l1_partial, so loss and gradient equal the
// separate entry points' bit for bit; kVec: planes of a multiple of 4 voxels and aligned volumes, by
// 16-byte accesses.
// As four kernels (profile, L1, its tree, factors) 16 us at 128^3, s = 2, and 33 us at 256 x 256 x 128, s
// = 4; here 9 and 27 us (151 MB). All 1,024 blocks of 128 threads are resident at once; with 256 threads
// and 3 (4) blocks per SM 12 and 32 (28) us; one LR voxel per thread with 4-byte accesses 9 and 48 us.
// (kS = 0: any number s_, I read again from the cache.) With more than four slices a thread's column is
// too long a chain where there are few LR voxels or no 16-byte accesses (61 x 45 x 37, s = 16: 22 us; 33
// x 33 x 256, s = 8: 14; 255 x 255 x 128, s = 8: 65); the step then takes profile, L1 and factors as
// three kernels (11, 12 and 39 us). 256 x 256 x 128: s = 5 37 in one, 35 in three; s = 8 30 and 33 (with
// the columns in registers 35).
constexpr int kFusedSlices = 4, kFusedSlicesVec = 8;
constexpr int64_t kFusedVoxels = 1 << 17;

static bool fused_profile(int s, int64_t n_lr, bool vec) {
    return s <= kFusedSlices || (vec && s >= kFusedSlicesVec && n_lr >= kFusedVoxels);
}

template <int kS, bool kVec>
__global__ void __launch_bounds__(kL1Threads, 7) k_profile_loss(
    const float* __restrict__ Iv, const float* __restrict__ Wv, const float* __restrict__ target, unsigned plane,
    FastDiv by_plane, int64_t n_lr, int64_t n_hr, int s_, float inv_s, float inv_n, float eps,
    float* __restrict__ lr_pred, float2* __restrict__ aip, float* partials, int* ticket, float* loss,
    StepCount count) {
    pdl_enter();
    count_step(count);
    constexpr int kV = kVec ? 4 : 1;  // consecutive LR voxels taken at once
    const int s = kS > 0 ? kS : s_;
    const int64_t t0 = int64_t(blockIdx.x) * kL1Threads + threadIdx.x;
    float acc = 0.f;
    for (int64_t q = 4 * t0; q < n_lr; q += 4 * kL1Blocks * kL1Threads) {
#pragma unroll
        for (int64_t i = q; i < q + 4; i += kV) {
            if (i >= n_lr) break;
            const unsigned k = fast_div(static_cast<unsigned>(i), by_plane);
            // first HR voxel of the column: (k s) plane + (i - k plane)
            const int64_t v0 = i + int64_t(k) * (s - 1) * plane;
            Voxels<kV> col[kS > 0 ? kS : 1], sum = {}, g;
#pragma unroll
            for (int j = 0; j < s; ++j) {
                const Voxels<kV> x = load_voxels<kV>(Iv + v0 + int64_t(j) * plane);
                if (kS > 0) col[kS > 0 ? j : 0] = x;
#pragma unroll
                for (int e = 0; e < kV; ++e) sum.v[e] += x.v[e];
            }
            const Voxels<kV> t = load_voxels<kV>(target + i);
#pragma unroll
            for (int e = 0; e < kV; ++e) {
                // (the profile's mean rounds before the difference, as when it is stored)
                const float d = __fmul_rn(sum.v[e], inv_s) - t.v[e];
                acc += fabsf(d);
                g.v[e] = l1_sign(d, inv_n);
            }
            store_voxels<kV>(lr_pred + i, g);
#pragma unroll
            for (int j = 0; j < s; ++j) {
                const int64_t v = v0 + int64_t(j) * plane;
                const Voxels<kV> w = load_voxels<kV>(Wv + v);
                const Voxels<kV> x = kS > 0 ? col[kS > 0 ? j : 0] : load_voxels<kV>(Iv + v);
                float2 a[kV];
#pragma unroll
                for (int e = 0; e < kV; ++e) a[e] = adj_factor(g.v[e] * inv_s, w.v[e], x.v[e], eps);
                if constexpr (kV == 4) {
                    reinterpret_cast<float4*>(aip + v)[0] = make_float4(a[0].x, a[0].y, a[1].x, a[1].y);
                    reinterpret_cast<float4*>(aip + v)[1] = make_float4(a[2].x, a[2].y, a[3].x, a[3].y);
                } else {
                    aip[v] = a[0];
                }
            }
        }
    }
    for (int64_t v = n_lr * s + t0; v < n_hr; v += kL1Blocks * kL1Threads)
        aip[v] = adj_factor(0.f, Wv[v], Iv[v], eps);
    l1_finish(acc, inv_n, partials, ticket, loss);
}

// Blocks of up to 256 threads over a plane's pieces (whole warps where there are 32 or more), the rest
// over the slices; about 32 blocks per SM, so few large planes and many small ones fill the chip too: a
// grid of at most 64 blocks per slice with all threads along the plane took 185 us where 27 are enough (4
// planes of 2,047 x 2,047, s = 4) and 52 in place of 7 (100,000 planes of one voxel).
struct Grid2d {
    dim3 grid, block;
};

static Grid2d grid2d(int64_t per_plane, int64_t slices) {
    unsigned tx = 1;
    if (per_plane < 32)
        while (tx < per_plane) tx *= 2;
    else
        tx = per_plane < 256 ? static_cast<unsigned>((per_plane + 31) / 32 * 32) : 256;
    const unsigned ty = 256 / tx;
    const int64_t by = slices < 1 ? 1 : (slices + ty - 1) / ty, gy = by < 65535 ? by : 65535;
    const int64_t bx = (per_plane + tx - 1) / tx, most = kSms * 32 / gy > 64 ? kSms * 32 / gy : 64;
    return {dim3(static_cast<unsigned>(bx < most ? bx : most), static_cast<unsigned>(gy)), dim3(tx, ty)};
}

static bool vec_ok(const void* a, const void* b, int64_t plane) {
    return plane % 4 == 0 && aligned16(a) && aligned16(b);
}

// The mean's normaliser: n, or n_norm > 0 when these values are one part of a larger mean.
static float l1_inv_n(int64_t n, int64_t n_norm) {
    const int64_t nn = n_norm > 0 ? n_norm : n;
    return nn > 0 ? 1.0f / float(nn) : 0.0f;
}

static gs_status launch_l1(const float* pred, const float* target, int64_t n, float* d_loss, float* dpred,
                    float* partials, cudaStream_t st, int64_t n_norm, int* ticket, const StepCount& count) {
    const float inv_n = l1_inv_n(n, n_norm);
    const bool vec = aligned16(pred) && aligned16(target) && (!dpred || aligned16(dpred));
    launch_k(vec ? k_l1_partial<true> : k_l1_partial<false>, dim3(kL1Blocks), dim3(kL1Threads), 0, st, pred,
        target, n, inv_n, dpred, partials, ticket, d_loss, count);
    gs_status s = last_launch_status();
    if (s != GS_OK || ticket) return s;
    launch_k(k_l1_final, dim3(1), dim3(kL1Threads), 0, st, partials, inv_n, d_loss);
    return last_launch_status();
}

template <bool kVec>
static gs_status launch_profile_loss(const float* I, const float* W, const float* target, int nz, int ny, int nx,
                                     int s, float eps, float* lr_pred, float* d_loss, int64_t n_norm,
                                     const Workspace& ws, const StepCount& count, cudaStream_t st) {
    const int64_t plane = int64_t(ny) * nx, n_lr = plane * (nz / s);
    auto go = [&](auto kernel) {
        launch_k(kernel, dim3(kL1Blocks), dim3(kL1Threads), 0, st, I, W, target, static_cast<unsigned>(plane),
            make_fastdiv(static_cast<unsigned>(plane)), n_lr, plane * nz, s, 1.0f / float(s),
            l1_inv_n(n_lr, n_norm), eps, lr_pred, ws.aip, ws.l1_part, ws.ticket, d_loss, count);
    };
    switch (s) {
        case 1: go(k_profile_loss<1, kVec>); break;
        case 2: go(k_profile_loss<2, kVec>); break;
        case 3: go(k_profile_loss<3, kVec>); break;
        case 4: go(k_profile_loss<4, kVec>); break;
        default:
            if constexpr (kVec) go(k_profile_loss<0, true>);  // (fused_profile)
    }
    return last_launch_status();
}

gs_status downsample_fwd_impl(const float* hr, int nz, int ny, int nx, int s, float* lr,
                              cudaStream_t st) {
    const int nzl = nz / s;
    const int64_t plane = int64_t(ny) * nx;
    if (nzl == 0) return GS_OK;
    const bool vec = vec_ok(hr, lr, plane);
    const Grid2d g = grid2d(vec ? plane / 4 : plane, nzl);
    auto go = [&](auto kernel) {
        launch_k(kernel, g.grid, g.block, 0, st, hr, static_cast<unsigned>(plane), static_cast<unsigned>(nzl), s,
            1.0f / float(s), lr);
    };
    switch (s) {
        case 1: vec ? go(k_downsample_fwd<4, 1>) : go(k_downsample_fwd<1, 1>); break;
        case 2: vec ? go(k_downsample_fwd<4, 2>) : go(k_downsample_fwd<1, 2>); break;
        case 3: vec ? go(k_downsample_fwd<4, 3>) : go(k_downsample_fwd<1, 3>); break;
        case 4: vec ? go(k_downsample_fwd<4, 4>) : go(k_downsample_fwd<1, 4>); break;
        case 5: vec ? go(k_downsample_fwd<4, 5>) : go(k_downsample_fwd<1, 5>); break;
        case 6: vec ? go(k_downsample_fwd<4, 6>) : go(k_downsample_fwd<1, 6>); break;
        case 7: vec ? go(k_downsample_fwd<4, 7>) : go(k_downsample_fwd<1, 7>); break;
        case 8: vec ? go(k_downsample_fwd<4, 8>) : go(k_downsample_fwd<1, 8>); break;
        default: vec ? go(k_downsample_fwd<4, 0>) : go(k_downsample_fwd<1, 0>);
    }
    return last_launch_status();
}

gs_status downsample_bwd_impl(const float* dlr, int nz, int ny, int nx, int s, float* dhr,
                              cudaStream_t st) {
    const int nzl = nz / s;
    const int64_t plane = int64_t(ny) * nx;
    const bool vec = vec_ok(dlr, dhr, plane);
    const Grid2d g = grid2d(vec ? plane / 4 : plane, nzl + (nz > nzl * s ? 1 : 0));
    launch_k(vec ? k_downsample_bwd<4> : k_downsample_bwd<1>, g.grid, g.block, 0, st, dlr, nz,
        static_cast<unsigned>(plane), static_cast<unsigned>(nzl), s, 1.0f / float(s), dhr);
    return last_launch_status();
}

static gs_status launch_profile_factors(const float* dlr, int nz, int ny, int nx, int s, const float* I, const float* W,
                                        float eps, float2* aip, cudaStream_t st) {
    const int64_t plane = int64_t(ny) * nx;
    const bool vec = vec_ok(I, W, plane) && aligned16(dlr);
    const Grid2d g = grid2d(vec ? plane / 4 : plane, nz);
    launch_k(vec ? k_profile_factors<4> : k_profile_factors<1>, g.grid, g.block, 0, st, dlr, static_cast<unsigned>(nz),
        static_cast<unsigned>(plane), static_cast<unsigned>(nz / s), static_cast<unsigned>(s), 1.0f / float(s), I, W,
        eps, aip);
    return last_launch_status();
}

// Provided by the other translation units.
gs_status bind_workspace(void* base, size_t bytes, int64_t n_gauss, int64_t capacity,
                         const gs_grid* grid, const gs_config* cfg, Workspace* ws);
bool bins_match(const gs_bins* b, const gs_grid* grid, const gs_config* cfg);
bool adam_ok(const gs_adam* hp);
gs_status bin_bricks_impl(const float* params, const gs_grid* grid, const gs_config* cfg,
                          gs_bins* bins, const Workspace& ws, cudaStream_t st);
gs_status render_fwd_impl(const gs_bins* bins, const gs_grid* grid, const gs_config* cfg, float* I,
                          float* W, unsigned long long* stats, cudaStream_t st);
gs_status launch_adjoint_pairs(const gs_bins* bins, const gs_grid* grid, const gs_config* cfg,
                               const Workspace& ws, cudaStream_t st);
gs_status launch_chain_adam(float* params, float* grad, float* m, float* v, const float* part,
                            const float* gacc, const gs_bins* bins, int64_t n,
                            const gs_grid* grid, const gs_config* cfg, const gs_adam* hp,
                            const int32_t* d_step, cudaStream_t st);

}  // namespace gs

using namespace gs;

static bool vol_args_ok(const void* a, const void* b, int32_t nz, int32_t ny, int32_t nx, int32_t s) {
    return a && b && nz > 0 && ny > 0 && nx > 0 && s > 0 &&
           int64_t(nz) * ny * nx <= (int64_t(1) << 31) - 1;
}

extern "C" gs_status gs_downsample_fwd(const float* hr, int32_t nz, int32_t ny, int32_t nx,
                                       int32_t s, float* lr, gs_stream stream) {
    if (!vol_args_ok(hr, lr, nz, ny, nx, s)) return GS_ERR_INVALID_ARG;
    return downsample_fwd_impl(hr, nz, ny, nx, s, lr, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" gs_status gs_downsample_bwd(const float* dlr, int32_t nz, int32_t ny, int32_t nx,
                                       int32_t s, float* dhr, gs_stream stream) {
    if (!vol_args_ok(dlr, dhr, nz, ny, nx, s)) return GS_ERR_INVALID_ARG;
    return downsample_bwd_impl(dlr, nz, ny, nx, s, dhr, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" gs_status gs_l1_loss(const float* pred, const float* target, int64_t n, float* d_loss,
                                float* dpred, void* ws, size_t ws_bytes, gs_stream stream) {
    if (!pred || !target || !d_loss || !ws || n <= 0) return GS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(ws) % 256 != 0) return GS_ERR_INVALID_ARG;
    if (ws_bytes < sizeof(float) * kL1Blocks) return GS_ERR_WORKSPACE;
    return launch_l1(pred, target, n, d_loss, dpred, static_cast<float*>(ws),
                     reinterpret_cast<cudaStream_t>(stream), 0, nullptr, StepCount{});
}

namespace {

// One fitting iteration's common part: validation, workspace and phase events.
struct FitRun {
    gs_fit_state* st = nullptr;
    Workspace w = {};
    cudaStream_t cs = nullptr;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaEvent_t lr_ready = nullptr;  // if set: the LR target is ready when this event is

    // Phase events: during stream capture they must be external event-record nodes, or they
    // would only serve as capture-internal dependencies.
    bool mark(int phase) const {
        if (!st->n_phase_events) return true;
        cudaEvent_t ev = static_cast<cudaEvent_t>(st->phase_events[phase]);
        if (cap == cudaStreamCaptureStatusActive)
            return cudaEventRecordWithFlags(ev, cs, cudaEventRecordExternal) == cudaSuccess;
        return cudaEventRecord(ev, cs) == cudaSuccess;
    }
};

gs_status fit_prepare(gs_fit_state* st, gs_stream stream, FitRun* run) {
    if (!st) return GS_ERR_INVALID_ARG;
    gs_status s = validate_grid_cfg(&st->grid, &st->cfg);
    if (s != GS_OK) return s;
    if (st->n_gauss <= 0) return GS_ERR_INVALID_ARG;
    const bool trilinear = st->lr_model == GS_LR_TRILINEAR;
    if (trilinear) {
        const int32_t lim = 1 << 23;
        if (st->lr_nx <= 0 || st->lr_ny <= 0 || st->lr_nz <= 0 || st->lr_nx >= lim ||
            st->lr_ny >= lim || st->lr_nz >= lim || st->grid.nx >= lim || st->grid.ny >= lim ||
            st->grid.nz >= lim)
            return GS_ERR_INVALID_ARG;
    } else if (st->lr_model != GS_LR_ZBOX || st->s <= 0 || st->grid.nz / st->s <= 0) {
        return GS_ERR_INVALID_ARG;
    }
    if (!st->params || !st->grad || !st->m || !st->v || !st->d_step || !st->I || !st->W ||
        !st->lr_pred || !st->lr_target || !st->d_loss)
        return GS_ERR_INVALID_ARG;
    if (!bins_match(&st->bins, &st->grid, &st->cfg) || st->bins.n_gauss != st->n_gauss)
        return GS_ERR_INVALID_ARG;
    s = bind_workspace(st->ws, st->ws_bytes, st->n_gauss, st->bins.capacity, &st->grid, &st->cfg,
                       &run->w);
    if (s != GS_OK) return s;
    if (st->n_phase_events != 0 && (st->n_phase_events != GS_FIT_PHASES || !st->phase_events))
        return GS_ERR_INVALID_ARG;
    run->st = st;
    run->cs = reinterpret_cast<cudaStream_t>(stream);
    if (st->n_phase_events && cudaStreamIsCapturing(run->cs, &run->cap) != cudaSuccess)
        return GS_ERR_CUDA;
    return GS_OK;
}

// Bin, render, LR forward model, L1 (normalised by n_norm LR values when n_norm > 0, else by
// the state's own count), its adjoint with the adjoint render's per-voxel factors, and the
// adjoint render kernel; phase events 0-4. The loss kernel counts the step in d_step unless that is
// nullptr: the Adam kernel behind it reads the counter already advanced, and no launch is left that
// only counts.
gs_status fit_front(const FitRun& run, int64_t n_norm, int32_t* d_step) {
    gs_fit_state* st = run.st;
    const Workspace& w = run.w;
    cudaStream_t cs = run.cs;
    const bool trilinear = st->lr_model == GS_LR_TRILINEAR;
    const gs_grid& g = st->grid;
    const StepCount count{d_step, st->bins.d_npairs, st->bins.capacity};
    if (!run.mark(0)) return GS_ERR_CUDA;
    gs_status s = bin_bricks_impl(st->params, &g, &st->cfg, &st->bins, w, cs);
    if (s != GS_OK) return s;
    if (!run.mark(1)) return GS_ERR_CUDA;
    s = render_fwd_impl(&st->bins, &g, &st->cfg, st->I, st->W, nullptr, cs);
    if (s != GS_OK) return s;
    if (!run.mark(2)) return GS_ERR_CUDA;
    if (run.lr_ready && cudaStreamWaitEvent(cs, run.lr_ready, 0) != cudaSuccess) return GS_ERR_CUDA;
    if (trilinear) {
        s = resample_fwd_impl(st->I, g.nz, g.ny, g.nx, st->lr_pred, st->lr_nz, st->lr_ny, st->lr_nx, cs);
        if (s != GS_OK) return s;
        const int64_t n_lr = int64_t(st->lr_nz) * st->lr_ny * st->lr_nx;
        // L1 loss; its gradient overwrites lr_pred in place.
        s = launch_l1(st->lr_pred, st->lr_target, n_lr, st->d_loss, st->lr_pred, w.l1_part, cs, n_norm, w.ticket,
                      count);
        if (s != GS_OK) return s;
        s = resample_adj_prep_impl(st->lr_pred, st->lr_nz, st->lr_ny, st->lr_nx, st->I, st->W, g.nz,
                                   g.ny, g.nx, st->cfg.eps, w.aip, cs);
    } else {
        const int64_t n_lr = int64_t(g.nz / st->s) * g.ny * g.nx;
        const bool vec = vec_ok(st->I, st->W, int64_t(g.ny) * g.nx) && aligned16(st->lr_target) &&
                         aligned16(st->lr_pred);
        if (fused_profile(st->s, n_lr, vec)) {
            s = (vec ? launch_profile_loss<true> : launch_profile_loss<false>)(
                st->I, st->W, st->lr_target, g.nz, g.ny, g.nx, st->s, st->cfg.eps, st->lr_pred, st->d_loss, n_norm,
                w, count, cs);
        } else {
            s = downsample_fwd_impl(st->I, g.nz, g.ny, g.nx, st->s, st->lr_pred, cs);
            if (s != GS_OK) return s;
            s = launch_l1(st->lr_pred, st->lr_target, n_lr, st->d_loss, st->lr_pred, w.l1_part, cs, n_norm, w.ticket,
                          count);
            if (s != GS_OK) return s;
            s = launch_profile_factors(st->lr_pred, g.nz, g.ny, g.nx, st->s, st->I, st->W, st->cfg.eps, w.aip, cs);
        }
    }
    if (s != GS_OK) return s;
    if (!run.mark(3)) return GS_ERR_CUDA;
    s = launch_adjoint_pairs(&st->bins, &g, &st->cfg, w, cs);
    if (s != GS_OK) return s;
    if (!run.mark(4)) return GS_ERR_CUDA;
    return GS_OK;
}

}  // namespace

extern "C" gs_status gs_fit_step(gs_fit_state* st, gs_stream stream) {
    FitRun run;
    gs_status s = fit_prepare(st, stream, &run);
    if (s != GS_OK) return s;
    if (!adam_ok(&st->adam)) return GS_ERR_INVALID_ARG;  // before the loss kernel counts the step
    s = fit_front(run, 0, st->d_step);
    if (s != GS_OK) return s;
    s = launch_chain_adam(st->params, st->grad, st->m, st->v, run.w.part, run.w.gacc, &st->bins,
                          st->n_gauss, &st->grid, &st->cfg, &st->adam, st->d_step, run.cs);
    if (s != GS_OK) return s;
    if (!run.mark(5)) return GS_ERR_CUDA;
    if (!run.mark(6)) return GS_ERR_CUDA;
    return GS_OK;
}

namespace {

// Per-device side stream and events of gs_fit_step_host, created once with that device current.
struct HostCopyRes {
    cudaStream_t side = nullptr;
    cudaEvent_t entry = nullptr, lr_done = nullptr;
};
constexpr int kMaxHostDevices = 64;
std::mutex g_host_res_mutex;
HostCopyRes g_host_res[kMaxHostDevices];

gs_status host_copy_res(HostCopyRes** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxHostDevices) return GS_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_host_res_mutex);
    HostCopyRes& r = g_host_res[dev];
    if (!r.side) {
        if (cudaStreamCreateWithFlags(&r.side, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&r.entry, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&r.lr_done, cudaEventDisableTiming) != cudaSuccess)
            return GS_ERR_CUDA;
    }
    *out = &r;
    return GS_OK;
}

}  // namespace

extern "C" gs_status gs_fit_step_host(gs_fit_state* st, const float* h_params,
                                      const float* h_lr_target, float* h_loss, gs_stream stream) {
    if (!st || st->n_gauss <= 0 || !st->params || !st->lr_target || !st->d_loss)
        return GS_ERR_INVALID_ARG;
    cudaStream_t cs = reinterpret_cast<cudaStream_t>(stream);
    const int64_t n_lr = st->lr_model == GS_LR_TRILINEAR
                             ? int64_t(st->lr_nz) * st->lr_ny * st->lr_nx
                             : (st->s > 0 ? int64_t(st->grid.nz / st->s) * st->grid.ny * st->grid.nx : 0);
    if (n_lr <= 0) return GS_ERR_INVALID_ARG;
    FitRun run;
    gs_status s = fit_prepare(st, stream, &run);
    if (s != GS_OK) return s;
    if (!adam_ok(&st->adam)) return GS_ERR_INVALID_ARG;
    // The parameters go first, alone on the link, since binning waits for them; the LR target
    // follows on a side stream while the step bins and renders, and the step waits for it
    // only before the LR model. The side stream starts after everything issued on `stream`
    // so far (the parameter copy included), so an earlier step still reading lr_target is
    // not overwritten.
    if (h_params && cudaMemcpyAsync(st->params, h_params, sizeof(float) * 12 * st->n_gauss,
                                    cudaMemcpyHostToDevice, cs) != cudaSuccess)
        return GS_ERR_CUDA;
    if (h_lr_target) {
        HostCopyRes* r = nullptr;
        s = host_copy_res(&r);
        if (s != GS_OK) return s;
        if (cudaEventRecord(r->entry, cs) != cudaSuccess ||
            cudaStreamWaitEvent(r->side, r->entry, 0) != cudaSuccess ||
            cudaMemcpyAsync(const_cast<float*>(st->lr_target), h_lr_target, sizeof(float) * n_lr,
                            cudaMemcpyHostToDevice, r->side) != cudaSuccess ||
            cudaEventRecord(r->lr_done, r->side) != cudaSuccess)
            return GS_ERR_CUDA;
        run.lr_ready = r->lr_done;
    }
    s = fit_front(run, 0, st->d_step);
    if (s != GS_OK) return s;
    s = launch_chain_adam(st->params, st->grad, st->m, st->v, run.w.part, run.w.gacc, &st->bins,
                          st->n_gauss, &st->grid, &st->cfg, &st->adam, st->d_step, cs);
    if (s != GS_OK) return s;
    if (!run.mark(5) || !run.mark(6)) return GS_ERR_CUDA;
    if (h_loss && cudaMemcpyAsync(h_loss, st->d_loss, sizeof(float), cudaMemcpyDeviceToHost,
                                  cs) != cudaSuccess)
        return GS_ERR_CUDA;
    return GS_OK;
}

extern "C" gs_status gs_fit_grad(gs_fit_state* st, int64_t n_lr_total, gs_stream stream) {
    if (n_lr_total < 0) return GS_ERR_INVALID_ARG;
    FitRun run;
    gs_status s = fit_prepare(st, stream, &run);
    if (s != GS_OK) return s;
    s = fit_front(run, n_lr_total, nullptr);
    if (s != GS_OK) return s;
    s = launch_chain_grad(st->params, st->grad, run.w.part, run.w.gacc, &st->bins, st->n_gauss,
                          &st->grid, &st->cfg, run.cs);
    if (s != GS_OK) return s;
    if (!run.mark(5)) return GS_ERR_CUDA;
    if (!run.mark(6)) return GS_ERR_CUDA;
    return GS_OK;
}

extern "C" gs_status gs_fit_apply(gs_fit_state* st, const int32_t* d_skip, gs_stream stream) {
    if (!st || st->n_gauss <= 0 || !st->params || !st->grad || !st->m || !st->v || !st->d_step)
        return GS_ERR_INVALID_ARG;
    return launch_adam(st->params, st->grad, st->m, st->v, st->n_gauss, &st->adam, st->d_step,
                       d_skip, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" gs_status gs_status_read(const int32_t* d_status, int32_t* h_status, gs_stream stream) {
    if (!d_status || !h_status) return GS_ERR_INVALID_ARG;
    cudaStream_t cs = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(h_status, d_status, sizeof(int32_t), cudaMemcpyDeviceToHost, cs) != cudaSuccess)
        return GS_ERR_CUDA;
    if (cudaStreamSynchronize(cs) != cudaSuccess) return GS_ERR_CUDA;
    if (*h_status & GS_STATUS_CAPACITY) return GS_ERR_CAPACITY;
    if (*h_status & GS_STATUS_NONFINITE) return GS_ERR_NONFINITE;
    return GS_OK;
}

extern "C" const char* gs_status_string(gs_status s) {
    switch (s) {
        case GS_OK: return "ok";
        case GS_ERR_INVALID_ARG: return "invalid argument";
        case GS_ERR_CAPACITY: return "pair capacity exceeded";
        case GS_ERR_WORKSPACE: return "workspace too small";
        case GS_ERR_CUDA: return "CUDA error";
        case GS_ERR_TIMEOUT: return "device wait timed out";
        case GS_ERR_NONFINITE: return "invalid Gaussian parameters";
    }
    return "unknown status";
}

extern "C" unsigned long long gs_launch_count(void) { return g_launches.load(); }

extern "C" const char* gs_version(void) { return "gsmri 0.1.0 (sm_103a)"; }

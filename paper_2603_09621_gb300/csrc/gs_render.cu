// gs_render.cu -- Eq. 3-4 forward render and its Eq. 5-6 adjoint, one CTA per brick (Sec. 3.3: "each
// handled by one CUDA thread block"; the brick's Gaussians are staged into shared memory and no depth
// order is needed).
//
// Exponent of a pair (voxel p, Gaussian i) in voxel units: q = S(dy, dz) + (sa (dx - dx*))^2 (record
// layout in gs_common.cuh), the Gaussian kernel is 2^-q and the pair contributes only where q <= T =
// (log2 e / 2) trunc_sigma^2. q is computed by the same operation sequence in both kernels from the
// voxel's global index and the Gaussian alone, so forward and adjoint agree on every inclusion decision
// and no result depends on the brick shape.
//
// Forward: the brick is split into 4 x 4 x 4 footprints, a quarter-warp each (a half or a whole warp in
// bricks of two or one); a lane owns the two x-rows of four (two, one) voxels at z and z + 1. The block
// stages the brick's list in rounds of 20 records per footprint (160 for an 8^3 brick); smaller bricks,
// with shorter lists, take shorter rounds (64 records for one or two footprints) and keep more blocks
// resident. The thread that stages a record tests it against every footprint (three conservative tests,
// see foot_mask: the triangle inequality in whitened space |M (p - mu)| >= |M (c - mu)| - rho4, with rho4
// the whitened radius of the footprint around its centre c; the truncated ellipsoid's bounding box
// widened by 3/2 along each axis; and q's lower bound from the smallest eigenvalue at the footprint's
// nearest point; a margin absorbs FP32 rounding). Each warp lists the hits of its footprints and
// evaluates them in ascending Gaussian id, accumulating S and W in registers (deterministic; one packed
// FFMA2 updates a voxel's (S, W) with (v r, r) g).
// Adjoint: one thread per (brick, Gaussian) pair evaluates the brick rows the Gaussian reaches (the row
// shadow, per z-row a quadratic in dy; z-planes whose section of the ellipsoid misses the brick's x range
// are skipped), each row as bx predicated voxel slots in packed FP32x2 pairs, so lanes never diverge
// inside a row. A block takes 256 consecutive brick-major pairs (one to three bricks), computes their row
// masks and counting-sorts them by number of rows in shared memory; its four warps then take 32-pair
// chunks of the sorted list, longest first, from a shared counter, so the lanes of a warp run pairs of
// equal length and a warp that drew short pairs moves on to the next chunk (64 registers without spills,
// 8 blocks per SM, 7 for 16-voxel-wide bricks; the y and z cross moments are summed over both FP32x2
// elements per row to keep the accumulators that small). The per-voxel factors (alpha, alpha I'), alpha =
// dL/dI / max(W, eps), are precomputed into one float2 volume; a block copies those of its first four
// bricks into shared memory (zero outside the grid), so rows read them without range tests; a 16-byte pad
// after every 128 bytes and a 32-byte offset between staged bricks spread the rows that the lanes of a
// warp read at once over the shared-memory banks. Each pair's partial is summed by one thread in a fixed
// voxel order (the processing order does not change results) and goes to a per-pair slot (deterministic
// mode, reduced later in Gaussian-major order) or to three vector atomics of four floats (fast mode).
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "gs_common.cuh"

namespace gs {

constexpr int kFwdChunkPerFoot = 20;  // Gaussians staged per forward round and 4^3 footprint (80 or 160 records)
constexpr int kFwdChunkSmall = 64;    // and for bricks of one or two footprints (see k_render_fwd)
constexpr int kBwdThreads = 128;
constexpr int kBwdPairs = 256;        // pairs per adjoint block, taken by warps 32 at a time
constexpr int kBwdStage = 4;          // bricks of per-voxel factors staged per adjoint block
constexpr int kMaxBrickVoxels = 512;  // brick volume limit (x * y * z <= 512)

// Packed FP32x2 arithmetic (one FFMA2 / FADD2 / FMUL2 instruction for two single-precision
// operations; each element is rounded exactly as the scalar fmaf / + / *).
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

struct RenderGeo {
    int nx, ny, nz;
    int bsx, bsy, bsz;  // brick shape
    int fx, fy, fz;     // 4^3 footprints per brick along each axis
    int nbx, nby;
    int bsy_shift, bsy_mask;  // row r of a brick is (y, z) = (r & mask, r >> shift)
    float T;            // (log2 e / 2) trunc_sigma^2: a pair contributes when q <= T
    float Tcull;        // cull bound on q: T (1 + 1e-2) + 1e-3
    float sqrtTcull;    // sqrt(Tcull)
    float eps;
    FastDiv dnbx, dnby;  // division by the brick counts along x and y
};

// Brick coordinates (along x, y, z) of brick index b (x fastest).
__device__ __forceinline__ void brick_xyz(int b, const RenderGeo& G, int& bx, int& by, int& bz) {
    const unsigned q = fast_div(static_cast<unsigned>(b), G.dnbx);
    bx = b - static_cast<int>(q) * G.nbx;
    const unsigned r = fast_div(q, G.dnby);
    by = static_cast<int>(q - r * static_cast<unsigned>(G.nby));
    bz = static_cast<int>(r);
}

struct Rec {
    float nmhx, nmlx;        // minus the mean's x head and tail
    float2 nmh_yz, nml_yz;   // minus the mean's (y, z) head and tail
    float2 pc2;              // (P2yz, c2): the dz coefficients of the row terms
    float2 pyc1;             // (Pyy, c1): their dy coefficients
    float pzz, sa, rho4, vr, r, v;
    float lam;               // q per squared voxel distance from the mean, at the least (culling)
    float ex, ey, ez;        // footprint-centre box half-extents (culling)
};

__device__ __forceinline__ Rec load_rec(const float4* s) {
    const float4 a = s[0], b = s[1], c = s[2], d = s[3], e = s[4];
    Rec R;
    R.nmhx = a.x; R.nmlx = a.y; R.nmh_yz = make_float2(a.z, a.w);
    R.nml_yz = make_float2(b.x, b.y); R.pc2 = make_float2(b.z, b.w);
    R.pyc1 = make_float2(c.x, c.y); R.pzz = c.z; R.sa = c.w;
    R.rho4 = d.y;
    R.ex = d.x; R.ey = d.z; R.ez = d.w;
    R.vr = e.x; R.r = e.y; R.v = e.z; R.lam = e.w;
    return R;
}

// The adjoint's copy of a record: quads 0, 1, 2 and 4 (it never reads quad 3, the footprint
// radius). Slots keep the full 80-byte stride: a 64-byte stride puts the pairs' quads into
// two bank groups and the shared-memory loads conflict.
__device__ __forceinline__ Rec load_rec_bwd(const float4* s) {
    const float4 a = s[0], b = s[1], c = s[2], e = s[4];
    Rec R;
    R.nmhx = a.x; R.nmlx = a.y; R.nmh_yz = make_float2(a.z, a.w);
    R.nml_yz = make_float2(b.x, b.y); R.pc2 = make_float2(b.z, b.w);
    R.pyc1 = make_float2(c.x, c.y); R.pzz = c.z; R.sa = c.w;
    R.rho4 = 0.f;
    R.ex = R.ey = R.ez = 0.f;
    R.vr = e.x; R.r = e.y; R.v = e.z; R.lam = 0.f;
    return R;
}

// Row quantities of the Gaussian for the row through voxel centres (., y, z): the row shadow
// S and the position dx* of the row minimum. One operation sequence for both kernels.
__device__ __forceinline__ void row_terms(const Rec& R, float2 fyz, float& dy, float& dz,
                                          float& S, float& dxs) {
    // (dy, dz) = ((y, z) - head) - tail as one packed pair of additions of the negated mean
    const float2 d = add2(add2(fyz, R.nmh_yz), R.nml_yz);
    dy = d.x;
    dz = d.y;
    // (Pyy dy + P2yz dz, c1 dy + c2 dz) as one packed multiply and one packed FMA
    const float2 t = fma2(R.pyc1, f2(dy, dy), mul2(R.pc2, f2(dz, dz)));
    S = fmaf(dy, t.x, R.pzz * dz * dz);
    dxs = t.y;
}

// x offset of voxel x from the mean, u = ux_base(R, x & ~3) + (x & 3).
__device__ __forceinline__ float ux_base(const Rec& R, int x4) {
    return (float(x4) + R.nmhx) + R.nmlx;
}

// The scaled x offset of voxel x = x4 + k (x4 = x & ~3) from the row minimum, tq = sa (u - dx*),
// is taken as tq = fma(k, sa, tq0) from the group's tq0 = sa (ux_base(R, x4) - dx*); then
// q = fma(tq, tq, S). Both kernels use this operation sequence, so forward and adjoint agree
// on every inclusion q <= T.

// Footprint cull: bit f of the result is set where the Gaussian of the record may reach a voxel
// centre of the brick's 4^3 footprint f = (wz FY + wy) FX + wx. Three conservative tests per
// footprint, at its centre (half-width 3/2 per axis): the whitened triangle inequality; the
// centre's offset from the mean against the truncated ellipsoid's box widened by the half-width;
// and q's lower bound lam |p - mu|^2 at the footprint's nearest point (exact for isotropic
// Gaussians, it drops footprints that only a corner of the ellipsoid grazes between voxel
// centres). (An approximate square root suffices: Tcull carries a 1 % margin over T.)
// kFX, kFY, kFZ: footprints per axis at compile time (0: taken from G).
template <int kFX, int kFY, int kFZ>
__device__ __forceinline__ unsigned foot_mask(const Rec& R, const RenderGeo& G, int ox, int oy, int oz) {
    const int fx = kFX > 0 ? kFX : G.fx, fy = kFY > 0 ? kFY : G.fy, fz = kFZ > 0 ? kFZ : G.fz;
    unsigned mask = 0;
    int bit = 0;
#pragma unroll (kFZ > 0 ? kFZ : 1)
    for (int wz = 0; wz < fz; ++wz)
#pragma unroll (kFY > 0 ? kFY : 1)
        for (int wy = 0; wy < fy; ++wy) {
            float dy, dz, S, dxs;
            row_terms(R, f2(float(oy + 4 * wy) + 1.5f, float(oz + 4 * wz) + 1.5f), dy, dz, S, dxs);
            const float ay = fmaxf(fabsf(dy) - 1.5f, 0.0f), az = fmaxf(fabsf(dz) - 1.5f, 0.0f);
            const float ayz = fmaf(ay, ay, az * az);
            const bool in_yz = (fabsf(dy) <= R.ey) & (fabsf(dz) <= R.ez);
#pragma unroll (kFX > 0 ? kFX : 1)
            for (int wx = 0; wx < fx; ++wx, ++bit) {
                const float ux = (float(ox + 4 * wx) + 1.5f + R.nmhx) + R.nmlx;
                const float tq = R.sa * (ux - dxs);
                const float qc = fmaf(tq, tq, S);
                const float ax = fmaxf(fabsf(ux) - 1.5f, 0.0f);
                const bool hit = (sqrt_approx(fmaxf(qc, 0.0f)) - R.rho4 <= G.sqrtTcull) & (fabsf(ux) <= R.ex) &
                                 in_yz & (R.lam * fmaf(ax, ax, ayz) <= G.sqrtTcull * G.sqrtTcull);
                mask |= hit ? 1u << bit : 0u;
            }
        }
    return mask;
}

// ------------------------------------------------------------------------ forward

// One block of 32 or 64 threads per brick (more with kFew, below). What bounds it is instruction issue
// (72 % active) and the latency of the gathered records, so work per instruction decides:
//   - A quarter-warp per 4^3 footprint, a lane owning the x-rows at z and z + 1: the row terms, offsets
//     and exponents of the two rows run as FP32x2 pairs (element by element the scalar operations, so
//     results are bit-identical to one row per lane). Against a half-warp per footprint and one row per
//     lane: 277 -> 241 us (256 x 256 x 128 grid, 500k Gaussians of a fit in progress, 132M effective
//     pairs, L2 flushed), 6.97 -> 6.13 ms (512 x 512 x 256 grid, 4M clustered Gaussians).
//   - The thread that stages a record also culls it against all the brick's footprints from registers
//     (row terms shared along x). With one lane per (record, footprint) reading the staged copy, the
//     cull's shared-memory loads were half of all its wavefronts, and staging and culling took 110 us of
//     the 241. Each warp then lists its footprints' hits of the whole round, so quarters of unequal hit
//     counts wait for one another once per round instead of once per 32 records: 241 -> 215 us, 6.13 ->
//     5.28 ms.
//   - Four hits per iteration (the lists are padded with a null record): 215 -> 212 us, 5.28 -> 5.17 ms,
//     and 35 -> 27 us where few bricks leave one warp per scheduler (32^3 grid, 4,096 Gaussians). Two
//     hits 217 us, eight 215 us.
//   - 72 registers, 14 blocks per SM, 20 records per round and footprint: 209 us and 5.23 ms. 16 records
//     212 us and 5.20 ms; 24 records 207 us but 5.50 ms; 64 registers (spills) 216 us; 96 registers 217
//     us. Rounds double-buffered with cp.async measured slower (242 against 241 us, 7.06 against 6.13
//     ms).
// kLanes: lanes per footprint, 8 as above; 16 in bricks of two footprints and 32 in bricks of one, which
// would leave half or three quarters of the only warp idle. Rounds of 64 records there fill the staging
// passes of 32. Random clouds on 128^3, against a quarter-warp and rounds of 40: 8 x 4 x 4 bricks 193 ->
// 142 us, 4^3 314 -> 202 (a half-warp per footprint throughout took 146 and 221; rounds of 32 or 96: 148
// and 205, 151 and 209).
// A grid of few bricks leaves most schedulers with one warp or none, and a brick's time is the latency of
// its lists. There (kFew) a footprint gets a whole warp, each lane the two voxels at z and z + 1, and a
// thread fetches its record of the next round while the present one is evaluated. Forward us, narrow ->
// whole warps: 8 bricks of 8^3 25 -> 21, 64 bricks 33-38 -> 26-28 (random and clustered clouds), 216
// bricks 35-46 -> 34-36, but 512 bricks 41-53 -> 51-56 and 4,096 bricks 146 -> 270: a lane with one voxel
// per row repeats the row terms four times as often. 8 x 8 x 4 bricks: 128 of them 36-42 -> 24-26, 1,024
// 43-64 -> 48-54. So where all footprints' warps are resident at once (152 SMs of 2 blocks of 8 warps:
// 304 bricks of 8^3, 608 of 8 x 8 x 4; bricks of one footprint have two warps, for staging). Eight hits
// per iteration 1-2 us slower.
constexpr int64_t kFewFootprints = kSms * 16;
constexpr int kFwdHits = 4;  // hits per iteration of the evaluation loop (one 32-bit list word)

template <bool kStats, int kChunk, int kLanes, bool kFew>
__global__ void __launch_bounds__(kFew ? 256 : 64, kFew ? 2 : 14) k_render_fwd(const int32_t* __restrict__ brick_off,
                                                       const int32_t* __restrict__ pair_gid,
                                                       const float4* __restrict__ rec4, RenderGeo G,
                                                       float* __restrict__ I, float* __restrict__ W,
                                                       unsigned long long* __restrict__ stats) {
    pdl_enter();
    static_assert(kChunk < 256, "hit lists hold record slots in bytes");
    // quads 0, 1, 2 and 4 of each record; slot kChunk is the null record (v r = r = 0: it adds 0)
    __shared__ float4 srec[4][kChunk + 1];
    __shared__ unsigned char sfoot[kChunk];
    __shared__ __align__(4) unsigned char slist[8][kChunk + kFwdHits];
    const int tid = threadIdx.x, lane = tid & 31;
    const int nthreads = blockDim.x;
    const int b = blockIdx.x;
    int bx, by, bz;
    brick_xyz(b, G, bx, by, bz);
    // kLanes lanes per 4^3 footprint, a lane owns kX voxels from lx on of two x-rows, at z and z + 1
    static_assert(kLanes == 8 || kLanes == 16 || kLanes == 32, "a lane owns 4, 2 or 1 voxels of a row");
    constexpr int kFoot = 32 / kLanes;  // footprints per warp
    constexpr int kX = 32 / kLanes;
    const int foot = tid / kLanes, foot0 = (tid >> 5) * kFoot;
    const int lx = (lane % (kLanes / 8)) * kX, lyz = (lane % kLanes) / (kLanes / 8);
    const int n_foot = G.fx * G.fy * G.fz;
    const bool foot_ok = foot < n_foot;
    const int f = foot_ok ? foot : 0;
    const int wx = f % G.fx, wy = (f / G.fx) % G.fy, wz = f / (G.fx * G.fy);
    const int x0 = bx * G.bsx, y0 = by * G.bsy, z0 = bz * G.bsz;
    const int ox = x0 + wx * 4, oy = y0 + wy * 4, oz = z0 + wz * 4;
    const int y = oy + (lyz & 3), z = oz + 2 * (lyz >> 2);
    const float fy = float(y);
    const float2 fz2 = f2(float(z), float(z + 1));
    if (tid < 4) srec[tid][kChunk] = make_float4(0.f, 0.f, 0.f, 0.f);

    float2 SWa[kX], SWb[kX];  // (S, W) of the lane's voxels in its two rows
#pragma unroll
    for (int xi = 0; xi < kX; ++xi) SWa[xi] = SWb[xi] = f2(0.f, 0.f);
    unsigned long long n_eff = 0, n_eval = 0;
    const int start = brick_off[b], end = brick_off[b + 1];
    // kFew: a thread stages at most one record per round, loaded while the round before is evaluated
    float4 qw[kFew ? REC_F4 : 1];
    auto fetch = [&](int gid, float4 (&q)[REC_F4]) {
        const float4* src = rec4 + int64_t(gid) * REC_F4;
#pragma unroll
        for (int part = 0; part < REC_F4; ++part) q[part] = src[part];
    };
    auto put = [&](int k, const float4 (&q)[REC_F4]) {
        const Rec R = load_rec(q);
        const unsigned m = (G.fx == 2 && G.fy == 2 && G.fz == 2) ? foot_mask<2, 2, 2>(R, G, x0, y0, z0)
                           : (G.fx == 2 && G.fy == 2 && G.fz == 1)
                               ? foot_mask<2, 2, 1>(R, G, x0, y0, z0)
                               : foot_mask<0, 0, 0>(R, G, x0, y0, z0);
        sfoot[k] = static_cast<unsigned char>(m);
        srec[0][k] = q[0];
        srec[1][k] = q[1];
        srec[2][k] = q[2];
        srec[3][k] = q[4];
    };
    int gid = start + tid < end ? pair_gid[start + tid] : 0;  // the thread's next record
    if constexpr (kFew) {
        if (start + tid < end && tid < kChunk) fetch(gid, qw);
    }
    for (int c0 = start; c0 < end; c0 += kChunk) {
        const int cnt = min(kChunk, end - c0);
        if (c0 != start) __syncthreads();  // the previous chunk's records are no longer read
        if constexpr (kFew) {
            if (tid < cnt) put(tid, qw);
        } else {
            for (int k = tid; k < cnt; k += nthreads) {
                float4 q[REC_F4];
                const int next = k + nthreads < cnt ? pair_gid[c0 + k + nthreads] : 0;
                fetch(gid, q);
                put(k, q);
                gid = next;
            }
        }
        __syncthreads();
        if (c0 + kChunk + tid < end) gid = pair_gid[c0 + kChunk + tid];
        if constexpr (kFew) {
            if (c0 + kChunk + tid < end && tid < kChunk) fetch(gid, qw);
        }
        // each warp lists the hits of its footprints in ascending Gaussian id
        int n[kFoot] = {};
        for (int k0 = 0; k0 < cnt; k0 += 32) {
            const int k = k0 + lane;
            const unsigned m = (k < cnt ? static_cast<unsigned>(sfoot[k]) : 0u) >> foot0;
#pragma unroll
            for (int j = 0; j < kFoot; ++j) {
                const unsigned bal = __ballot_sync(0xffffffffu, (m >> j) & 1u);
                if ((m >> j) & 1u)
                    slist[foot0 + j][n[j] + __popc(bal & ((1u << lane) - 1u))] = static_cast<unsigned char>(k);
                n[j] += __popc(bal);
            }
        }
        int myn = n[0];
        if constexpr (kFoot == 4)
            myn = (lane & 16) ? ((lane & 8) ? n[3] : n[2]) : ((lane & 8) ? n[1] : n[0]);
        else if constexpr (kFoot == 2)
            myn = (lane & 16) ? n[1] : n[0];
        if (lyz < kFwdHits && lx == 0) slist[foot][myn + lyz] = static_cast<unsigned char>(kChunk);
        __syncwarp();
        for (int i = 0; i < myn; i += kFwdHits) {
            const unsigned slots = *reinterpret_cast<const unsigned*>(&slist[foot][i]);
#pragma unroll
            for (int u = 0; u < kFwdHits; ++u) {
                const int kk = (slots >> (8 * u)) & 0xff;
                const float4 ra = srec[0][kk], rb = srec[1][kk], rc = srec[2][kk], re = srec[3][kk];
                const float dy = (fy + ra.z) + rb.x;
                const float2 dz = add2(add2(fz2, f2(ra.w, ra.w)), f2(rb.y, rb.y));
                const float2 dy2 = f2(dy, dy);
                const float2 t = fma2(f2(rc.x, rc.x), dy2, mul2(f2(rb.z, rb.z), dz));
                const float2 dxs = fma2(f2(rc.y, rc.y), dy2, mul2(f2(rb.w, rb.w), dz));
                const float2 Sr = fma2(dy2, t, mul2(mul2(f2(rc.z, rc.z), dz), dz));
                const float ux = (float(ox) + ra.x) + ra.y;
                const float2 sa2 = f2(rc.w, rc.w);
                const float2 tq0 = mul2(sa2, add2(f2(ux, ux), f2(-dxs.x, -dxs.y)));
                const float2 vrr = f2(re.x, re.y);
#pragma unroll
                for (int xi = 0; xi < kX; ++xi) {
                    // (k = 0 in the packed FMA gives tq0 itself)
                    const float k = float(lx + xi);
                    const float2 tq = (kX == 4 && xi == 0) ? tq0 : fma2(f2(k, k), sa2, tq0);
                    const float2 q = fma2(tq, tq, Sr);
                    if (q.x <= G.T) {
                        const float g = ex2_approx(-q.x);
                        SWa[xi] = fma2(vrr, f2(g, g), SWa[xi]);
                    }
                    if (q.y <= G.T) {
                        const float g = ex2_approx(-q.y);
                        SWb[xi] = fma2(vrr, f2(g, g), SWb[xi]);
                    }
                    if (kStats) {
                        const bool live = i + u < myn;
                        const bool in = live && y < G.ny && ox + lx + xi < G.nx;
                        n_eff += (in && z < G.nz && q.x <= G.T) ? 1 : 0;
                        n_eff += (in && z + 1 < G.nz && q.y <= G.T) ? 1 : 0;
                        n_eval += live ? 2 : 0;
                    }
                }
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!(foot_ok && y < G.ny && z + h < G.nz)) continue;
        const int64_t row = (int64_t(z + h) * G.ny + y) * G.nx + ox + lx;
        float Iv[kX], Wv[kX];
#pragma unroll
        for (int xi = 0; xi < kX; ++xi) {
            const float S = h ? SWb[xi].x : SWa[xi].x;
            Wv[xi] = h ? SWb[xi].y : SWa[xi].y;
            Iv[xi] = S / (Wv[xi] > G.eps ? Wv[xi] : G.eps);
        }
        if constexpr (kX == 4) {
            if (ox + 3 < G.nx && (G.nx & 3) == 0) {
                store4<true>(I + row, Iv);
                store4<true>(W + row, Wv);
                continue;
            }
        }
#pragma unroll
        for (int xi = 0; xi < kX; ++xi)
            if (ox + lx + xi < G.nx) {
                I[row + xi] = Iv[xi];
                W[row + xi] = Wv[xi];
            }
    }
    if (kStats) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            n_eff += __shfl_xor_sync(0xffffffffu, n_eff, o);
            n_eval += __shfl_xor_sync(0xffffffffu, n_eval, o);
        }
        if (lane == 0) {
            atomicAdd(&stats[0], n_eff);
            atomicAdd(&stats[1], n_eval);
        }
    }
}

// ------------------------------------------------------------------------ adjoint

// Rows of the brick (index rz * bsy + ry) that the Gaussian may reach: per z-row the row
// shadow S(dy, dz) <= Tcull holds on the y-interval yc(dz) +- hw(dz), with
// yc = mu_y - (P2yz / 2 Pyy) dz and hw^2 = Tcull / Pyy - c3 dz^2,
// c3 = (Pzz - P2yz^2 / 4 Pyy) / Pyy (the interval is padded; Tcull carries a 1 % margin).
// A z-plane whose section of the truncated ellipsoid misses the brick's x range is skipped, and the
// interval of a section that passes the brick's nearer x face is cut where it does: 13 % fewer rows on
// a fit's cloud, 23 % on clustered ones, for 15 instructions more per plane; backward call 378 -> 373 us
// (256 x 256 x 128 / 500k), 7.59 -> 7.46 ms (512 x 512 x 256 / 4M clustered).
// The mask is a conservative superset only (the rows themselves test q <= T), so the plane
// offsets are taken as dz(z0) + rz and positions relative to the brick, inside the padding.
// kBY, kBZ: the brick's y and z sizes at compile time (0: taken from G); the fitting
// workload's 8^3 bricks and the paper's 8 x 8 x 4 ones have their own unrolled copies.
template <int kBY, int kBZ>
__device__ __forceinline__ unsigned long long brick_row_mask(const Rec& R, const RenderGeo& G,
                                                             int x0, int y0, int z0) {
    const int bsy = kBY > 0 ? kBY : G.bsy;
    const int bsz = kBZ > 0 ? kBZ : G.bsz;
    unsigned long long mask = 0;
    const float ipyy = __fdividef(1.0f, R.pyc1.x);
    const float k1 = -0.5f * (R.pc2.x * ipyy);
    const float nc3 = -(R.pzz - 0.25f * R.pc2.x * (R.pc2.x * ipyy)) * ipyy;
    const float h0 = fminf(G.Tcull * ipyy, 1e37f);  // (finite: 3e18 voxels, for a Tcull without bound, reach any row)
    const float mu_y = -(R.nmh_yz.x + R.nml_yz.x);
    const float mu_x = -(R.nmhx + R.nmlx);
    const float pad = 1e-3f + 1e-5f * fabsf(mu_y);
    // the section's x extent through plane dz: centre mu_x + (c1 k1 + c2) dz, half-width
    // hw_y lam, lam^2 = Pyy / a + c1^2 (hw_y the y half-width of the same section); tested as
    // |centre - brick centre| <= half-width + brick half-width
    const float kx = fmaf(R.pyc1.y, k1, R.pc2.y);
    const float beta2 = R.pyc1.x * __fdividef(1.0f, R.sa * R.sa);
    const float lam2 = fmaf(R.pyc1.y, R.pyc1.y, beta2);
    const float lam = sqrt_approx(lam2);
    const float il2 = __fdividef(1.0f, lam2);
    const float bl = sqrt_approx(beta2) * il2;
    const float half_bx = 0.5f * float(G.bsx - 1);
    const float xrel = mu_x - (float(x0) + half_bx);
    const float padx = 1e-3f + 1e-5f * fabsf(mu_x) + half_bx;
    const float yrel = mu_y - float(y0);
    const float dz0 = (float(z0) + R.nmh_yz.y) + R.nml_yz.y;
    const unsigned full = (1u << bsy) - 1u;
#pragma unroll (kBZ > 0 ? kBZ : 1)
    for (int rz = 0; rz < bsz; ++rz) {
        const float dz = dz0 + float(rz);
        const float hw2 = fmaf(nc3 * dz, dz, h0);
        // (1e-37: at 0 the product of root and reciprocal root is not a number)
        const float hw2b = fmaxf(hw2, 1e-37f);
        const float ish = rsqrt_approx(hw2b);
        const float sh = hw2b * ish;
        const float xc = fmaf(kx, dz, xrel);
        const bool in_x = fabsf(xc) <= fmaf(sh, lam, padx);
        // the section within the brick's nearer x face: at s = (y - yc) / hw its smallest |x| side is
        // |xc| + hw (c s - beta sqrt(1 - s^2)), c = sign(xc) c1, which meets the face at
        // s = (a c -+ beta sqrt(lam^2 - a^2)) / lam^2, a = (padx - |xc|) / hw; an end s = +-1 of the
        // section stays where it lies inside the face
        const float a = (padx - fabsf(xc)) * ish;
        const float c = __int_as_float(__float_as_int(R.pyc1.y) ^ (__float_as_int(xc) & 0x80000000));
        const float t = bl * sqrt_approx(fmaxf(fmaf(-a, a, lam2), 0.0f));
        const float e = a * c * il2;
        const float s1 = (c > a && e + t < 1.0f) ? e + t : 1.0f;
        const float s0 = (-c > a && e - t > -1.0f) ? e - t : -1.0f;
        const float yc = fmaf(k1, dz, yrel);
        const float ylo = fmaf(sh, s0, yc) - pad, yhi = fmaf(sh, s1, yc) + pad;
        // rows ceil(ylo) .. floor(yhi), clamped to the brick; empty when ia > ib
        const int ia = min(max(__float2int_ru(ylo), 0), bsy);
        const int ib = min(max(__float2int_rd(yhi), -1), bsy - 1);
        const unsigned bits = (full << ia) & (full >> (bsy - 1 - ib));
        if (hw2 >= 0.0f && in_x) mask |= static_cast<unsigned long long>(bits) << (rz * bsy);
    }
    return mask;
}

// Per-voxel adjoint factors (alpha, alpha I'): dL/dw_i = v_i alpha - alpha I' with
// alpha = dL/dI / max(W, eps) and I' = I where W > eps, else 0 (Eq. 5; below the floor
// I = S / eps, so dI/dw_i = v_i / eps).
// kVec: four voxels per thread by 16-byte accesses (aligned volumes), the last n mod 4 voxels by
// one thread each. Bound by HBM (20 bytes per voxel): one voxel per thread took 27 us at 4.7M
// voxels, 14 us now.
template <bool kVec>
__global__ void __launch_bounds__(256) k_bwd_prep(const float* __restrict__ Iv,
                                                  const float* __restrict__ Wv,
                                                  const float* __restrict__ dIv, int64_t n,
                                                  float eps, float2* __restrict__ aip) {
    pdl_enter();
    const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t step = int64_t(gridDim.x) * blockDim.x;
    if (kVec) {
        for (int64_t q = t; q < n / 4; q += step) {
            const float4 w = reinterpret_cast<const float4*>(Wv)[q];
            const float4 g = reinterpret_cast<const float4*>(dIv)[q];
            const float4 iv = reinterpret_cast<const float4*>(Iv)[q];
            const float2 a0 = adj_factor(g.x, w.x, iv.x, eps), a1 = adj_factor(g.y, w.y, iv.y, eps);
            const float2 a2 = adj_factor(g.z, w.z, iv.z, eps), a3 = adj_factor(g.w, w.w, iv.w, eps);
            reinterpret_cast<float4*>(aip)[2 * q] = make_float4(a0.x, a0.y, a1.x, a1.y);
            reinterpret_cast<float4*>(aip)[2 * q + 1] = make_float4(a2.x, a2.y, a3.x, a3.y);
        }
    }
    for (int64_t i = (kVec ? n / 4 * 4 : 0) + t; i < n; i += step)
        aip[i] = adj_factor(dIv[i], Wv[i], Iv[i], eps);
}

// Adjoint sums of one (brick, Gaussian) pair, with h = gamma g (gamma = dL/dw) per voxel.
// A brick row of bx voxels is taken as bx/2 voxel pairs (p, p + bx/2); element e of a float2
// holds the sums over the voxels p + e bx/2 (offset u = uc_e + p from the mean along x).
struct AdjAcc {
    float2 h, p1;         // sum h, sum h p
    float2 pq;            // sum h p (p + 1) / 2  (so sum h p^2 = 2 pq - p1)
    float2 ag;            // sum alpha g
    float hy, hz;         // sum h dy, sum h dz over both elements
    float oy, oz;         // sum h o dy, sum h o dz, o = p + e bx/2 the slot's offset from uc_0
    float yy, zz, yz;     // sum h dy^2, sum h dz^2, sum h dy dz
};

// The rows of one (brick, Gaussian) pair: for each row in the mask, bx voxel slots in bx/2
// packed pairs, with the factors read from the block's staged copy (kStaged: per row, float4
// (alpha_p, alpha_{p+bx/2}, -alpha I'_p, -alpha I'_{p+bx/2}) for p < bx/2) or from the volume.
// The exponent of every slot takes the forward's operation sequence element by element, so
// both kernels agree on every inclusion q <= T. The slot moments along x are running sums
// over p (descending), which need no per-slot constants.
template <int BX, bool kStaged>
__device__ __forceinline__ void adjoint_rows(const Rec& R, unsigned long long m, const RenderGeo& G,
                                             int x0, int y0, int z0,
                                             const float4* __restrict__ sfac_b,
                                             const float2* __restrict__ aip, AdjAcc& A) {
    constexpr int P = BX / 2;                    // voxel pairs per row
    constexpr int NT = (BX >= 8) ? BX / 8 : 1;   // packed group bases per row
    const int x1 = min(x0 + BX, G.nx) - 1;
    const float2 sa2 = f2(R.sa, R.sa), v2 = f2(R.v, R.v);
    // x offsets of the 4-voxel groups that pair p reads: (group p/4, group p/4 + bx/8)
    float2 uxp[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j)
        uxp[j] = (BX >= 8) ? f2(ux_base(R, x0 + 4 * j), ux_base(R, x0 + 4 * j + P))
                           : f2(ux_base(R, x0), ux_base(R, x0));
    while (m) {
        const int r = __ffsll(static_cast<long long>(m)) - 1;
        m &= m - 1;
        const int y = y0 + (r & G.bsy_mask), z = z0 + (r >> G.bsy_shift);
        float dy, dz, S, dxs;
        row_terms(R, f2(float(y), float(z)), dy, dz, S, dxs);
        const float2 S2 = f2(S, S), nd2 = f2(-dxs, -dxs);
        float2 tq0[NT];  // tq0 of each group, the forward's sa * (ux - dx*)
#pragma unroll
        for (int j = 0; j < NT; ++j) tq0[j] = mul2(sa2, add2(uxp[j], nd2));
        const bool row_in = kStaged || ((y < G.ny) && (z < G.nz));
        const float2* arow = kStaged ? nullptr
                                     : aip + (int64_t(min(z, G.nz - 1)) * G.ny + min(y, G.ny - 1)) * G.nx + x0;
        float2 rs = f2(0.f, 0.f), m1 = f2(0.f, 0.f), qs = f2(0.f, 0.f);
#pragma unroll
        for (int p = P - 1; p >= 0; --p) {
            // exponent of the two slots: in-group index k, group base tq0
            float2 tq;
            if (BX >= 8) {
                const int k = p & 3;
                tq = (k == 0) ? tq0[p >> 2] : fma2(f2(float(k), float(k)), sa2, tq0[p >> 2]);
            } else {
                tq = fma2(f2(float(p), float(p + 2)), sa2, tq0[0]);
            }
            const float2 q = fma2(tq, tq, S2);
            const float2 g = f2((q.x <= G.T) ? ex2_approx(-q.x) : 0.0f,
                                (q.y <= G.T) ? ex2_approx(-q.y) : 0.0f);
            float2 al, nai;  // (alpha, -alpha I') of the two slots, zero outside the grid
            if (kStaged) {
                const float4 f = sfac_b[r * P + ((r * P) >> 3) + p];
                al = f2(f.x, f.y);
                nai = f2(f.z, f.w);
            } else {
                const float2 fa = (row_in && x0 + p <= x1) ? arow[p] : f2(0.f, 0.f);
                const float2 fb = (row_in && x0 + p + P <= x1) ? arow[p + P] : f2(0.f, 0.f);
                al = f2(fa.x, fb.x);
                nai = f2(-fa.y, -fb.y);
            }
            const float2 h = mul2(fma2(v2, al, nai), g);
            A.ag = fma2(al, g, A.ag);
            rs = add2(rs, h);            // sum over slots >= p
            if (p >= 1) {
                m1 = add2(m1, rs);       // ends as sum h p
                qs = add2(qs, m1);       // ends as sum h p (p + 1) / 2
            }
        }
        A.h = add2(A.h, rs);
        A.p1 = add2(A.p1, m1);
        A.pq = add2(A.pq, qs);
        const float s0 = rs.x + rs.y;
        const float s1 = fmaf(float(P), rs.y, m1.x + m1.y);  // sum h o over the row
        A.hy = fmaf(s0, dy, A.hy);
        A.hz = fmaf(s0, dz, A.hz);
        A.oy = fmaf(s1, dy, A.oy);
        A.oz = fmaf(s1, dz, A.oz);
        const float ty = dy * s0;
        A.yy = fmaf(ty, dy, A.yy);
        A.yz = fmaf(ty, dz, A.yz);
        A.zz = fmaf(dz * s0, dz, A.zz);
    }
}

template <int BX, bool kDet>
__global__ void __launch_bounds__(kBwdThreads, (BX == 16 ? 7 : 8)) k_render_bwd(
    const int32_t* __restrict__ pair_gid, const int32_t* __restrict__ pair_gmj,
    const int32_t* __restrict__ pair_brick, const int64_t* __restrict__ npairs, int64_t capacity,
    const float4* __restrict__ rec4, RenderGeo G, const float2* __restrict__ aip,
    float* __restrict__ part, float* __restrict__ gacc) {
    pdl_enter();
    constexpr int kPer = kBwdPairs / kBwdThreads;  // pairs per thread in the prologue
    constexpr int kWarps = kBwdThreads / 32;
    // staged bricks 2 float4 apart beyond their padded size: rows of different bricks that the
    // lanes of a warp read at once fall on different banks
    constexpr int kStageStride = kMaxBrickVoxels / 2 + kMaxBrickVoxels / 16 + 2;
    __shared__ float4 sfac[kBwdStage * kStageStride];
    __shared__ unsigned long long smask[kBwdPairs];
    __shared__ int sgid[kBwdPairs];
    __shared__ unsigned short sorder[kBwdPairs];
    __shared__ unsigned char sstage[kBwdPairs];
    __shared__ int hist[66];
    __shared__ int cursor[66];
    __shared__ int sbrick[kBwdStage];
    __shared__ int gcount[kBwdPairs / 32];
    __shared__ int chunk_next;
    int64_t P = *npairs;
    if (P < 0 || P > capacity) P = 0;
    const int64_t base = int64_t(blockIdx.x) * kBwdPairs;
    if (base >= P) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nvalid = static_cast<int>(min(int64_t(kBwdPairs), P - base));
    for (int k = tid; k < 66; k += kBwdThreads) {
        hist[k] = 0;
        cursor[k] = 0;
    }
    if (tid == 0) chunk_next = 0;
    // distinct bricks of the block's pairs (brick-major order: a new brick starts a run);
    // thread tid holds pairs tid + h * 128 (32-pair group warp + 4 h)
    int b_t[kPer], gidv[kPer];
    unsigned bal[kPer];
    bool newb[kPer];
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
        const int q = tid + h * kBwdThreads;
        b_t[h] = 0;
        gidv[h] = 0;
        newb[h] = false;
        if (q < nvalid) {
            b_t[h] = pair_brick[base + q];
            gidv[h] = pair_gid[base + q];
            newb[h] = (q == 0) || (b_t[h] != pair_brick[base + q - 1]);
        }
        bal[h] = __ballot_sync(0xffffffffu, newb[h]);
        if (lane == 0) gcount[warp + h * kWarps] = __popc(bal[h]);
    }
    __syncthreads();
    int n_bricks = 0;
#pragma unroll
    for (int g = 0; g < kBwdPairs / 32; ++g) n_bricks += gcount[g];
    // row mask of each pair, its staged brick, histogram of row counts (most first)
    int bucket[kPer];
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
        const int q = tid + h * kBwdThreads;
        const int grp = warp + h * kWarps;
        bucket[h] = 0;
        if (q < nvalid) {
            int run_before = 0;
            for (int g = 0; g < grp; ++g) run_before += gcount[g];
            const int kb = run_before + __popc(bal[h] & ((1u << lane) - 1u)) + (newb[h] ? 1 : 0) - 1;
            if (newb[h] && kb < kBwdStage) sbrick[kb] = b_t[h];
            sstage[q] = static_cast<unsigned char>(min(kb, kBwdStage));
            const int gid = gidv[h];
            sgid[q] = gid;
            int bxx, by, bz;
            brick_xyz(b_t[h], G, bxx, by, bz);
            const Rec Rm = load_rec_bwd(rec4 + int64_t(gid) * REC_F4);
            const int mx0 = bxx * G.bsx, my0 = by * G.bsy, mz0 = bz * G.bsz;
            const unsigned long long m = (G.bsy == 8 && G.bsz == 8)
                                             ? brick_row_mask<8, 8>(Rm, G, mx0, my0, mz0)
                                             : (G.bsy == 8 && G.bsz == 4)
                                                   ? brick_row_mask<8, 4>(Rm, G, mx0, my0, mz0)
                                                   : brick_row_mask<0, 0>(Rm, G, mx0, my0, mz0);
            smask[q] = m;
            bucket[h] = 64 - __popcll(static_cast<long long>(m));
            atomicAdd(&hist[bucket[h]], 1);
        }
    }
    __syncthreads();
    if (warp == 0) {  // exclusive prefix of the 65 bucket counts: lane l owns buckets 3l..3l+2
        int c[3], t = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int bk = 3 * lane + k;
            c[k] = bk <= 64 ? hist[bk] : 0;
            t += c[k];
        }
        int incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int run = incl - t;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int bk = 3 * lane + k;
            if (bk <= 64) hist[bk] = run;
            run += c[k];
        }
    }
    // per-voxel factors of the first kBwdStage bricks into shared memory, zero outside the
    // grid, so the row loop needs no range tests; per row and voxel pair (p, p + bx/2) one
    // float4 (alpha_p, alpha_{p+bx/2}, -alpha I'_p, -alpha I'_{p+bx/2}), float4 index
    // i = row * bx/2 + p stored at i + i/8 (rows of the lanes of a warp fall on other banks)
    const int n_stage = min(n_bricks, kBwdStage);
    constexpr int kPairs = BX / 2;
    const int bpairs = kPairs * G.bsy * G.bsz;
    for (int k = 0; k < n_stage; ++k) {
        const int b = sbrick[k];
        int bxx, byy, bzz;
        brick_xyz(b, G, bxx, byy, bzz);
        const int x0 = bxx * BX, y0 = byy * G.bsy, z0 = bzz * G.bsz;
        float4* dst = &sfac[k * kStageStride];
        if (x0 + BX <= G.nx && y0 + G.bsy <= G.ny && z0 + G.bsz <= G.nz && (G.nx & 1) == 0) {
            // brick inside the grid, rows 16-byte aligned: float4 loads of voxels (2c, 2c+1)
            // and (2c+P, 2c+P+1) give the entries of pairs 2c and 2c+1
            constexpr int kHalf = kPairs / 2;
            for (int e = tid; e < bpairs / 2; e += kBwdThreads) {
                const int r = e / kHalf, c = e - r * kHalf;
                const int y = y0 + (r & G.bsy_mask), z = z0 + (r >> G.bsy_shift);
                const float2* src = aip + (int64_t(z) * G.ny + y) * G.nx + x0 + 2 * c;
                const float4 fa = *reinterpret_cast<const float4*>(src);
                const float4 fb = *reinterpret_cast<const float4*>(src + kPairs);
                dst[r * kPairs + ((r * kPairs) >> 3) + 2 * c] = make_float4(fa.x, fb.x, -fa.y, -fb.y);
                dst[r * kPairs + ((r * kPairs) >> 3) + 2 * c + 1] = make_float4(fa.z, fb.z, -fa.w, -fb.w);
            }
            continue;
        }
        for (int e = tid; e < bpairs; e += kBwdThreads) {
            const int r = e / kPairs, pp = e - r * kPairs;
            const int y = y0 + (r & G.bsy_mask), z = z0 + (r >> G.bsy_shift);
            const int xa = x0 + pp, xb = xa + kPairs;
            const float2* src = aip + (int64_t(min(z, G.nz - 1)) * G.ny + min(y, G.ny - 1)) * G.nx;
            const bool row_ok = y < G.ny && z < G.nz;
            const float2 fa = (row_ok && xa < G.nx) ? src[xa] : make_float2(0.f, 0.f);
            const float2 fb = (row_ok && xb < G.nx) ? src[xb] : make_float2(0.f, 0.f);
            dst[e + (e >> 3)] = make_float4(fa.x, fb.x, -fa.y, -fb.y);
        }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
        const int q = tid + h * kBwdThreads;
        if (q < nvalid)
            sorder[hist[bucket[h]] + atomicAdd(&cursor[bucket[h]], 1)] = static_cast<unsigned short>(q);
    }
    __syncthreads();
    // warps take 32-pair chunks of the sorted list (longest first) until none is left, so a
    // warp that drew short pairs goes on with the next chunk instead of idling
    const int nchunks = (nvalid + 31) / 32;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&chunk_next, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= nchunks) break;
        const int rank = c * 32 + lane;
        if (rank >= nvalid) continue;
        const int lt = sorder[rank];
        const int64_t i = base + lt;
        const unsigned long long m = smask[lt];
        if (m == 0ull) {
            // a pair whose Gaussian reaches none of the brick's rows (the count-sorted list puts
            // them in the last chunks): its partial is zero, with no record or brick to load
            if (kDet) {
                float4* dst = reinterpret_cast<float4*>(part + int64_t(pair_gmj[i]) * GRAD_FLOATS);
                const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
                dst[0] = z4;
                dst[1] = z4;
                dst[2] = z4;
            }
            continue;
        }
        const int b = pair_brick[i];
        int bx, by, bz;
        brick_xyz(b, G, bx, by, bz);
        const int x0 = bx * BX, y0 = by * G.bsy, z0 = bz * G.bsz;
        const int stage = sstage[lt];
        const Rec R = load_rec_bwd(rec4 + int64_t(sgid[lt]) * REC_F4);
        AdjAcc A;
        A.h = A.p1 = A.pq = A.ag = f2(0.f, 0.f);
        A.hy = A.hz = A.oy = A.oz = A.yy = A.zz = A.yz = 0.f;
        if (stage < kBwdStage)
            adjoint_rows<BX, true>(R, m, G, x0, y0, z0, &sfac[stage * kStageStride],
                                   aip, A);
        else
            adjoint_rows<BX, false>(R, m, G, x0, y0, z0, nullptr, aip, A);
        // moments about the mean: slot p of element e sits at u = uc_e + p along x
        const float uc0 = ux_base(R, x0);
        const float uc1 = (BX >= 8) ? ux_base(R, x0 + BX / 2) : uc0 + 2.0f;
        float m1x = fmaf(uc0, A.h.x, A.p1.x) + fmaf(uc1, A.h.y, A.p1.y);
        // sum h u^2 = uc^2 sum h + 2 uc sum h p + (2 pq - p1)
        float m2xx = fmaf(uc0, fmaf(uc0, A.h.x, 2.0f * A.p1.x), fmaf(2.0f, A.pq.x, -A.p1.x)) +
                     fmaf(uc1, fmaf(uc1, A.h.y, 2.0f * A.p1.y), fmaf(2.0f, A.pq.y, -A.p1.y));
        // (the y, z cross moments take slot o at uc_0 + o)
        float m2xy = fmaf(uc0, A.hy, A.oy);
        float m2xz = fmaf(uc0, A.hz, A.oz);
        float m1y = A.hy, m1z = A.hz;
        float m2yy = A.yy, m2zz = A.zz, m2yz = A.yz;
        const float dvp = A.ag.x + A.ag.y, dr = A.h.x + A.h.y;
        const float rr = R.r;
        const float dv = rr * dvp;
        m1x *= rr; m1y *= rr; m1z *= rr;
        m2xx *= rr; m2yy *= rr; m2zz *= rr; m2xy *= rr; m2xz *= rr; m2yz *= rr;
        if (kDet) {
            const int64_t j = pair_gmj[i];
            float4* dst = reinterpret_cast<float4*>(part + j * GRAD_FLOATS);
            dst[0] = make_float4(m1x, m1y, m1z, m2xx);
            dst[1] = make_float4(m2yy, m2zz, m2xy, m2xz);
            dst[2] = make_float4(m2yz, dv, dr, 0.f);
        } else {
            // three 16-byte vector reductions (48-byte slots of a 256-byte-aligned array) in place
            // of eleven scalar ones: 8.22 -> 7.63 ms for the backward call on the 512 x 512 x 256
            // grid with 4M clustered Gaussians (104M pairs), whose scattered reductions were
            // the kernel's largest store traffic
            float4* dst = reinterpret_cast<float4*>(gacc + int64_t(sgid[lt]) * GRAD_FLOATS);
            atomicAdd(dst, make_float4(m1x, m1y, m1z, m2xx));
            atomicAdd(dst + 1, make_float4(m2yy, m2zz, m2xy, m2xz));
            atomicAdd(dst + 2, make_float4(m2yz, dv, dr, 0.f));
        }
    }
}

// ------------------------------------------------------------------------ host side

RenderGeo make_geo(const gs_grid* grid, const gs_config* cfg) {
    BrickGeom b = brick_geom(grid, cfg);
    RenderGeo G;
    G.nx = grid->nx; G.ny = grid->ny; G.nz = grid->nz;
    G.bsx = b.bx; G.bsy = b.by; G.bsz = b.bz;
    G.fx = b.bx / 4; G.fy = b.by / 4; G.fz = b.bz / 4;
    G.bsy_shift = (b.by == 4) ? 2 : ((b.by == 8) ? 3 : 4);
    G.bsy_mask = b.by - 1;
    G.nbx = b.nbx; G.nby = b.nby;
    G.T = kHalfLog2e * cfg->trunc_sigma * cfg->trunc_sigma;
    G.Tcull = G.T * (1.0f + 1e-2f) + 1e-3f;
    G.sqrtTcull = sqrtf(G.Tcull);
    G.eps = cfg->eps;
    G.dnbx = make_fastdiv(static_cast<unsigned>(b.nbx));
    G.dnby = make_fastdiv(static_cast<unsigned>(b.nby));
    return G;
}

gs_status render_fwd_impl(const gs_bins* bins, const gs_grid* grid, const gs_config* cfg,
                          float* I, float* W, unsigned long long* stats, cudaStream_t st) {
    RenderGeo G = make_geo(grid, cfg);
    const int n_foot = G.fx * G.fy * G.fz;
    // records staged per round about in proportion to the footprints (the lists of smaller
    // bricks are shorter), so that smaller bricks keep more blocks resident
    const float4* rec4 = reinterpret_cast<const float4*>(bins->rec);
    const bool few = int64_t(bins->n_bricks) * (n_foot > 1 ? n_foot : 2) <= kFewFootprints;
    const int lanes = few || n_foot == 1 ? 32 : (n_foot == 2 ? 16 : 8);
    // (few: a thread per record of a round, so two warps also for a single footprint)
    const int threads = few && n_foot == 1 ? 64 : 32 * ((n_foot * lanes + 31) / 32);
    auto go = [&](auto kernel) {
        launch_k(kernel, dim3(bins->n_bricks), dim3(threads), 0, st, bins->brick_off, bins->pair_gid,
            rec4, G, I, W, stats);
    };
    auto pick = [&](auto chunk) {
        constexpr int kChunk = decltype(chunk)::value;
        if (few)
            stats ? go(k_render_fwd<true, kChunk, 32, true>) : go(k_render_fwd<false, kChunk, 32, true>);
        else if (n_foot > 2)
            stats ? go(k_render_fwd<true, kChunk, 8, false>) : go(k_render_fwd<false, kChunk, 8, false>);
        else if constexpr (kChunk == kFwdChunkSmall) {
            if (n_foot == 2)
                stats ? go(k_render_fwd<true, kChunk, 16, false>) : go(k_render_fwd<false, kChunk, 16, false>);
            else
                stats ? go(k_render_fwd<true, kChunk, 32, false>) : go(k_render_fwd<false, kChunk, 32, false>);
        }
    };
    if (n_foot >= 6)
        pick(std::integral_constant<int, 8 * kFwdChunkPerFoot>{});
    else if (n_foot >= 3)
        pick(std::integral_constant<int, 4 * kFwdChunkPerFoot>{});
    else
        pick(std::integral_constant<int, kFwdChunkSmall>{});
    return last_launch_status();
}

gs_status bind_workspace(void* base, size_t bytes, int64_t n_gauss, int64_t capacity,
                         const gs_grid* grid, const gs_config* cfg, Workspace* ws);
bool bins_match(const gs_bins* b, const gs_grid* grid, const gs_config* cfg);

gs_status launch_bwd_prep(const float* I, const float* W, const float* dI, const RenderGeo& G,
                          const Workspace& ws, cudaStream_t st) {
    const int64_t nv = int64_t(G.nx) * G.ny * G.nz;
    const bool vec = aligned16(I) && aligned16(W) && aligned16(dI);
    const int64_t pb = ((vec ? nv / 4 : nv) + 256) / 256;
    launch_k(vec ? k_bwd_prep<true> : k_bwd_prep<false>, dim3(static_cast<unsigned>(pb < 65536 ? pb : 65536)),
        dim3(256), 0, st, I, W, dI, nv, G.eps, ws.aip);
    return last_launch_status();
}

template <int BX, bool kDet>
static gs_status launch_bwd_pairs(const gs_bins* bins, const RenderGeo& G, const Workspace& ws,
                                  cudaStream_t st) {
    if (bins->capacity == 0) return GS_OK;
    const unsigned gb = static_cast<unsigned>((bins->capacity + kBwdPairs - 1) / kBwdPairs);
    const float4* rec4 = reinterpret_cast<const float4*>(bins->rec);
    launch_k(k_render_bwd<BX, kDet>, dim3(gb), dim3(kBwdThreads), 0, st, bins->pair_gid,
        bins->pair_gmj, bins->pair_brick, bins->d_npairs, bins->capacity, rec4, G, ws.aip,
        kDet ? ws.part : nullptr, kDet ? nullptr : ws.gacc);
    return last_launch_status();
}

// Adjoint render kernel over ws.aip (already prepared): per-pair partials (deterministic) or
// atomically accumulated ws.gacc (fast; zeroed here).
gs_status launch_adjoint_pairs(const gs_bins* bins, const gs_grid* grid, const gs_config* cfg,
                               const Workspace& ws, cudaStream_t st) {
    RenderGeo G = make_geo(grid, cfg);
    const int64_t N = bins->n_gauss;
    if (!cfg->deterministic && N > 0 &&
        cudaMemsetAsync(ws.gacc, 0, sizeof(float) * GRAD_FLOATS * N, st) != cudaSuccess)
        return GS_ERR_CUDA;
    const bool det = cfg->deterministic != 0;
    switch (G.bsx) {
        case 4: return det ? launch_bwd_pairs<4, true>(bins, G, ws, st) : launch_bwd_pairs<4, false>(bins, G, ws, st);
        case 8: return det ? launch_bwd_pairs<8, true>(bins, G, ws, st) : launch_bwd_pairs<8, false>(bins, G, ws, st);
        case 16: return det ? launch_bwd_pairs<16, true>(bins, G, ws, st) : launch_bwd_pairs<16, false>(bins, G, ws, st);
    }
    return GS_ERR_INVALID_ARG;
}

}  // namespace gs

using namespace gs;

extern "C" gs_status gs_render_fwd(const gs_bins* bins, const gs_grid* grid, const gs_config* cfg,
                                   float* I, float* W, unsigned long long* d_stats,
                                   gs_stream stream) {
    gs_status s = validate_grid_cfg(grid, cfg);
    if (s != GS_OK) return s;
    if (!bins_match(bins, grid, cfg) || !I || !W) return GS_ERR_INVALID_ARG;
    return render_fwd_impl(bins, grid, cfg, I, W, d_stats, reinterpret_cast<cudaStream_t>(stream));
}

namespace {

// A thread's page-locked word and event of each device, for reading a pair count back while later
// work of the stream runs on; given back when the thread ends.
constexpr int kMaxDevices = 64;

struct CountSlot {
    int64_t* host = nullptr;
    cudaEvent_t copied = nullptr;
    ~CountSlot() {
        if (copied) (void)cudaEventDestroy(copied);
        if (host) (void)cudaFreeHost(host);
    }
};

CountSlot* count_slot() {
    static thread_local CountSlot slots[kMaxDevices];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    CountSlot& s = slots[dev];
    if (!s.host && cudaMallocHost(reinterpret_cast<void**>(&s.host), sizeof(int64_t)) != cudaSuccess) {
        s.host = nullptr;
        return nullptr;
    }
    if (!s.copied && cudaEventCreateWithFlags(&s.copied, cudaEventDisableTiming) != cudaSuccess) {
        s.copied = nullptr;
        return nullptr;
    }
    return &s;
}

// Voxels up to which the forward is queued before the pairs are known to fit: if they do not, it
// writes 8 bytes per voxel in vain (about 40 us at this size), else the GPU does not idle while the host
// reads the count and launches it (about 15 us).
constexpr int64_t kSpeculateVoxels = int64_t(1) << 25;

}  // namespace

extern "C" gs_status gs_render_cloud(const float* params, const gs_grid* grid, const gs_config* cfg,
                                     gs_bins* bins, void* ws, size_t ws_bytes, float* I, float* W,
                                     unsigned long long* d_stats, int64_t* h_npairs, gs_stream stream) {
    if (!h_npairs || !I || !W) return GS_ERR_INVALID_ARG;
    gs_status s = gs_bin_bricks(params, grid, cfg, bins, ws, ws_bytes, stream);
    if (s != GS_OK) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    CountSlot* slot = count_slot();
    if (!slot ||
        cudaMemcpyAsync(slot->host, bins->d_npairs, sizeof(int64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaEventRecord(slot->copied, st) != cudaSuccess)
        return GS_ERR_CUDA;
    const bool early = int64_t(grid->nx) * grid->ny * grid->nz <= kSpeculateVoxels;
    if (early) s = render_fwd_impl(bins, grid, cfg, I, W, d_stats, st);
    if (cudaEventSynchronize(slot->copied) != cudaSuccess) return GS_ERR_CUDA;
    *h_npairs = *static_cast<volatile int64_t*>(slot->host);
    if (s != GS_OK) return s;
    if (*h_npairs > bins->capacity) return GS_ERR_CAPACITY;
    return early ? GS_OK : render_fwd_impl(bins, grid, cfg, I, W, d_stats, st);
}

extern "C" gs_status gs_render_bwd(const float* params, const gs_bins* bins, const gs_grid* grid,
                                   const gs_config* cfg, const float* I, const float* W,
                                   const float* dI, float* dparams, void* ws, size_t ws_bytes,
                                   gs_stream stream) {
    gs_status s = validate_grid_cfg(grid, cfg);
    if (s != GS_OK) return s;
    if (!bins_match(bins, grid, cfg) || !I || !W || !dI) return GS_ERR_INVALID_ARG;
    if (bins->n_gauss > 0 && (!params || !dparams)) return GS_ERR_INVALID_ARG;
    Workspace w;
    s = bind_workspace(ws, ws_bytes, bins->n_gauss, bins->capacity, grid, cfg, &w);
    if (s != GS_OK) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    s = launch_bwd_prep(I, W, dI, make_geo(grid, cfg), w, st);
    if (s != GS_OK) return s;
    s = launch_adjoint_pairs(bins, grid, cfg, w, st);
    if (s != GS_OK || bins->n_gauss == 0) return s;
    // (the reduction over a Gaussian's pairs and the chain to its raw parameters in one kernel; as
    // two, with the sums through memory, 42 us against 39 us at 375,000 Gaussians and 2.1M pairs)
    return launch_chain_grad(params, dparams, w.part, w.gacc, bins, bins->n_gauss, grid, cfg, st);
}

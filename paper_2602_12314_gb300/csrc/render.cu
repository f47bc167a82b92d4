// Query rendering Q = R_f(G, T) (Sec. III-B, Eq. render_query): the depth-ordered alpha
// blending of Eq. (alpha_blending) applied to the d-dimensional query vectors f_i, and its
// backward with respect to f.
//
// One CTA per 16x16 tile, in the forward and the backward; the tile's Gaussians are staged through
// shared memory in batches (mean, exponent coefficients/opacity, query as float4 rows), so every query
// row is read from L2/HBM once per tile and broadcast to the 256 pixels.  (The backward of the full
// blend runs one warp per strip of a tile.)
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.cuh"

namespace lat {
namespace {

// Staged form of one splat: exponent coefficients q = (-a/2, -b, -c/2, opacity) of the conic
// (a, b, c).
__device__ __forceinline__ float4 stage_splat(float4 co) {
    return make_float4(__fmul_rn(-0.5f, co.x), -co.y, __fmul_rn(-0.5f, co.z), co.w);
}

// The hi and lo BF16 terms of (x0, x1), packed: hi = bf16(x), lo = bf16(x - hi).
__device__ __forceinline__ void tc_split(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - hf.x, x1 - hf.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// alpha of a splat at a pixel centre, or -1 when the exponent is positive.  Every rounding
// is explicit (fused multiply-adds written out), so the forward and backward kernels take
// bit-identical decisions for the same inputs.
__device__ __forceinline__ float splat_alpha(float2 m, float4 q, float px, float py) {
    const float dx = __fsub_rn(m.x, px), dy = __fsub_rn(m.y, py);
    const float power = __fmaf_rn(dx, __fmaf_rn(q.x, dx, __fmul_rn(q.y, dy)), __fmul_rn(__fmul_rn(q.z, dy), dy));
    if (power > 0.0f) return -1.0f;
    return fminf(kAlphaMax, __fmul_rn(q.w, __expf(power)));
}

// a.xy += w v.xy
__device__ __forceinline__ void fma2(float& a0, float& a1, float w, float v0, float v1) {
    fma2(Pair(w), Pair(v0, v1), Pair(a0, a1)).get(a0, a1);
}

// splat_alpha of the pixels (px, -npy.x) and (px, -npy.y): the same operations, two at a time.
__device__ __forceinline__ void splat_alpha2(float2 m, float4 q, float px, Pair npy, float& a0, float& a1) {
    const Pair dx(__fsub_rn(m.x, px)), dy = add2(Pair(m.y), npy);
    float p0, p1;
    fma2(dx, fma2(Pair(q.x), dx, mul2(Pair(q.y), dy)), mul2(mul2(Pair(q.z), dy), dy)).get(p0, p1);
    mul2(Pair(q.w), Pair(__expf(p0), __expf(p1))).get(a0, a1);
    a0 = p0 > 0.0f ? -1.0f : fminf(kAlphaMax, a0);
    a1 = p1 > 0.0f ? -1.0f : fminf(kAlphaMax, a1);
}

// Pixels per thread of the forward: two (a tile is 128 threads), one at d = 64, where two pixels'
// accumulators alone would take 128 registers.
template <int DQ>
constexpr int fwd_px() {
    return DQ <= 32 ? 2 : 1;
}
template <int DQ>
constexpr int fwd_threads() {
    return kTilePixels / fwd_px<DQ>();
}
// Blocks per SM that the registers must leave room for: at d = 64 two of 256 threads (without the
// bound the compiler takes 154 to 178 registers, one block: 1296 x 968, 1M Gaussians, the whole view
// 1,022 us against 766).
template <int DQ>
constexpr int fwd_blocks() {
    return DQ == 64 ? 2 : 1;
}

constexpr int kBatch = 128;  // Gaussians staged per round

template <int DQ, bool FULL = false>
struct FwdSmem {
    float2 xy[kBatch];
    float4 co[kBatch];
    float4 f[kBatch][DQ / 4];
    float4 cz[FULL ? kBatch : 1];  // colour, depth
};

// The further channels of the full Stage I render: colours (N x 3) and camera depths (N) blended
// with the queries' weights into C (n x 3) and Z.
struct FullImages {
    const float* colours;
    const float* depth;
    float* C;
    float* Z;
};

// Front-to-back blend of one tile.  Bound by issue and by the shared-memory broadcasts of the staged
// rows: a thread blends two vertically adjacent pixels, so that each row read from shared memory
// meets two pixels' FMAs (packed two channels each) and the two transmittance chains overlap.
// The pixels' exponents and transmittances are taken with packed arithmetic, two pixels an
// instruction.  (1200 x 680, 600k Gaussians, d = 32: 186 us with one pixel per thread, 151 with two.)
template <int DQ, bool FULL = false>
__device__ __forceinline__ void render_fwd_tile(const TileJob& job, FwdSmem<DQ, FULL>& sm, const FullImages& full = {}) {
    constexpr int DV = DQ / 4, PX = fwd_px<DQ>(), NT = fwd_threads<DQ>();
    const int tile = job.tile;
    const int tx = tile % job.tiles_x, ty = tile / job.tiles_x;
    const int t = threadIdx.x;
    const int px = tx * kTile + t % kTile, py = ty * kTile + t / kTile * PX;
    const float fpx = (float)px;
    const Pair npy(-(float)py, -(float)(py + 1));
    const int2 range = job.ranges[tile];
    float4 acc[PX][DV], acz[PX];
    float T[PX];
    int count[PX];
    bool done[PX], out = true;
#pragma unroll
    for (int i = 0; i < PX; ++i) {
#pragma unroll
        for (int k = 0; k < DV; ++k) acc[i][k] = make_float4(0.f, 0.f, 0.f, 0.f);
        acz[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        T[i] = 1.0f;
        count[i] = 0;
        done[i] = !(px < job.W && py + i < job.H);
        out = out && done[i];
    }
    for (int start = range.x; start < range.y; start += kBatch) {
        if (__syncthreads_count(out) == NT) break;
        const int k = start + t;
        if (t < kBatch && k < range.y) {
            const int g = job.pair_ids[k];
            sm.xy[t] = job.xy[g];
            sm.co[t] = stage_splat(job.conic_opac[g]);
#pragma unroll
            for (int c = 0; c < DV; ++c) sm.f[t][c] = job.f[(size_t)g * DV + c];
            if (FULL)
                sm.cz[t] = make_float4(full.colours[3 * (size_t)g], full.colours[3 * (size_t)g + 1],
                                       full.colours[3 * (size_t)g + 2], full.depth[g]);
        }
        __syncthreads();
        const int cnt = min(kBatch, range.y - start);
        for (int j = 0; j < cnt && !out; ++j) {
            const float2 m = sm.xy[j];
            const float4 q = sm.co[j];
            float w[PX], alphas[PX], left[PX];
            bool use[PX], any = false;
            if (PX == 2) {
                splat_alpha2(m, q, fpx, npy, alphas[0], alphas[PX - 1]);
                const Pair t2(T[0], T[PX - 1]), a2(alphas[0], alphas[PX - 1]);
                mul2(t2, add2(Pair(1.0f), Pair(-alphas[0], -alphas[PX - 1]))).get(left[0], left[PX - 1]);
                mul2(a2, t2).get(w[0], w[PX - 1]);
            } else {
                alphas[0] = splat_alpha(m, q, fpx, (float)py);
                left[0] = __fmul_rn(T[0], __fsub_rn(1.0f, alphas[0]));
                w[0] = __fmul_rn(alphas[0], T[0]);
            }
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                const float alpha = alphas[i], test_T = left[i];
                use[i] = !done[i] && !(alpha < kAlphaMin);
                if (use[i] && test_T < kTMin) {
                    done[i] = true;
                    use[i] = false;
                }
                if (use[i]) {
                    T[i] = test_T;
                    ++count[i];
                }
                any = any || use[i];
            }
            if (any) {
#pragma unroll
                for (int c = 0; c < DV; ++c) {
                    const float4 v = sm.f[j][c];
#pragma unroll
                    for (int i = 0; i < PX; ++i)
                        if (use[i]) {
                            fma2(acc[i][c].x, acc[i][c].y, w[i], v.x, v.y);
                            fma2(acc[i][c].z, acc[i][c].w, w[i], v.z, v.w);
                        }
                }
                if (FULL) {
                    const float4 v = sm.cz[j];
#pragma unroll
                    for (int i = 0; i < PX; ++i)
                        if (use[i]) {
                            fma2(acz[i].x, acz[i].y, w[i], v.x, v.y);
                            fma2(acz[i].z, acz[i].w, w[i], v.z, v.w);
                        }
                }
            }
            out = done[0] && done[PX - 1];
        }
    }
#pragma unroll
    for (int i = 0; i < PX; ++i)
        if (px < job.W && py + i < job.H) {
            const size_t p = (size_t)(py + i) * job.W + px;
#pragma unroll
            for (int c = 0; c < DV; ++c) job.Q[p * DV + c] = acc[i][c];
            if (FULL) {
                full.C[3 * p] = acz[i].x;
                full.C[3 * p + 1] = acz[i].y;
                full.C[3 * p + 2] = acz[i].z;
                full.Z[p] = acz[i].w;
            }
            job.T_final[p] = T[i];
            job.n_contrib[p] = count[i];
        }
}

template <int DQ>
__global__ void __launch_bounds__(fwd_threads<DQ>(), fwd_blocks<DQ>())
    render_fwd_kernel(CamParams cam, const int2* __restrict__ ranges, const int32_t* __restrict__ pair_ids,
                      const float2* __restrict__ xy, const float4* __restrict__ conic_opac,
                      const float4* __restrict__ f, float4* __restrict__ Q, float* __restrict__ T_final,
                      int32_t* __restrict__ n_contrib) {
    __shared__ FwdSmem<DQ> sm;
    const int tile = cam.tile_order ? cam.tile_order[blockIdx.x] : (int)blockIdx.x;
    const TileJob job{tile, cam.tiles_x, cam.W, cam.H, ranges, pair_ids, xy, conic_opac, f, Q, T_final, n_contrib,
                      nullptr, nullptr};
    render_fwd_tile<DQ>(job, sm);
}

// Next (frame, tile) of a batch from the global work list (frame in the top 12 bits), taken in
// list order by an atomic ticket; -1 when the list is exhausted.  Every thread returns the same
// item; the two barriers also keep the previous item's shared memory until every thread is done.
__device__ __forceinline__ int next_item(int* counter, const int32_t* order, int total) {
    __shared__ int s_item;
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
    __syncthreads();
    const int it = s_item;
    __syncthreads();
    return it < total ? order[it] : -1;
}

// Persistent render forward over every tile of every frame of a batch, longest lists first.  (At
// d = 32 held to five blocks per SM: over six 640 x 480 frames 475 us a launch against 492 at the
// four that its registers would allow; the single frame above is shorter with four, 57 against
// 70 us at 640 x 480, where the last tiles' own length counts.)
template <int DQ>
__global__ void __launch_bounds__(fwd_threads<DQ>(), DQ == 32 ? 5 : fwd_blocks<DQ>())
    render_fwd_batch_kernel(const __grid_constant__ BatchJobs jobs, const int32_t* __restrict__ order, int total,
                            int* __restrict__ counter) {
    __shared__ FwdSmem<DQ> sm;
    for (int item = next_item(counter, order, total); item >= 0; item = next_item(counter, order, total)) {
        TileJob job = jobs.fr[item >> 20];
        job.tile = item & 0xFFFFF;
        render_fwd_tile<DQ>(job, sm);
    }
}

// Backward of the query blend, df_i = sum_p w_ip dQ_p, as one small GEMM per tile and batch on
// the tensor cores: the weights w_ip of a batch of kBwdBatch Gaussians are first recomputed front
// to back by the pixel threads (the forward's arithmetic, so the same contributions are taken: a
// pixel stops after its n_contrib-th one) into a shared-memory matrix W^T (Gaussians x pixels),
// each weight as two BF16 terms w = hi + lo (hi = bf16(w), lo = bf16(w - hi)); the tile's dQ
// rows are held the same way.  Then warp (m, h) takes Gaussians 16m..16m+15 and channel half h
// and sums over the tile's 256 pixels with mma.sync m16n8k16 (BF16 in, FP32 accumulate) as
// W_hi dQ_hi + W_hi dQ_lo + W_lo dQ_hi (each product within 2^-16 of the FP32 one), and each
// non-zero (Gaussian, channel) sum goes to df with one atomic per tile.  A per-tile contraction
// of 64 x 256 x d does not amortise TMEM allocation and completion waits; the warp-level MMA
// runs in the registers of the warps that computed the weights.  Bound by the serial weight chains
// between the three barriers of a batch (848 x 480, 200k Gaussians, d = 32: 74 us).  A warp per
// 16 x 4 strip without block barriers, whose sums left as 16-byte atomics, took 48 us there and
// stopped with a misaligned address on other scenes (20,000 splats of about 27 pixels at 640 x 480;
// room keyframes at d = 64), although every index and address it formed was in bounds and aligned.
constexpr int kBwdBatch = 64;
constexpr int kWtStride = kTilePixels + 8;  // bf16 per W^T row (528 B: ldmatrix rows on distinct banks)

template <int DQ>
constexpr int dq_stride() {
    return DQ + 8;  // bf16 per dQ row (16 B of padding: ldmatrix rows on distinct banks)
}

template <int DQ>
constexpr size_t render_bwd_smem() {
    // W^T hi / lo, dQ hi / lo, staged splats
    return 2 * sizeof(__nv_bfloat16) * (size_t)kBwdBatch * kWtStride +
           2 * sizeof(__nv_bfloat16) * (size_t)kTilePixels * dq_stride<DQ>() +
           (sizeof(float4) + sizeof(float2) + sizeof(int)) * kBwdBatch;
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_trans(uint32_t addr, uint32_t (&r)[2]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
// c += a b, m16n8k16, BF16 operands, FP32 accumulators
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Backward of one tile (256 threads); smem is the dynamic shared memory of render_bwd_smem.
template <int DQ>
__device__ __forceinline__ void render_bwd_tile(const TileJob& job, float4* smem) {
    constexpr int DV = DQ / 4;
    constexpr int DQS = dq_stride<DQ>();
    constexpr int NT = DQ / 16;  // n-tiles of 8 channels per warp (a warp covers DQ / 2 channels)
    using bf16 = __nv_bfloat16;
    bf16* wt_hi = reinterpret_cast<bf16*>(smem);      // [Gaussian][pixel]
    bf16* wt_lo = wt_hi + (size_t)kBwdBatch * kWtStride;
    bf16* dq_hi = wt_lo + (size_t)kBwdBatch * kWtStride;  // [pixel][channel]
    bf16* dq_lo = dq_hi + (size_t)kTilePixels * DQS;
    float4* s_co = reinterpret_cast<float4*>(dq_lo + (size_t)kTilePixels * DQS);
    float2* s_xy = reinterpret_cast<float2*>(s_co + kBwdBatch);
    int* s_id = reinterpret_cast<int*>(s_xy + kBwdBatch);
    static_assert(((size_t)kBwdBatch * kWtStride * 2 * 2 + (size_t)kTilePixels * DQS * 2 * 2) % 16 == 0,
                  "staged splats stay 16-byte aligned");

    const int tile = job.tile;
    const int tx = tile % job.tiles_x, ty = tile / job.tiles_x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int px = tx * kTile + (t % kTile), py = ty * kTile + (t / kTile);
    const bool inside = px < job.W && py < job.H;
    const float fpx = (float)px, fpy = (float)py;
    const int2 range = job.ranges[tile];
    int remaining = 0;
    {
        // this pixel's dQ row as hi / lo terms
        float4 g[DV];
        if (inside) {
            const size_t p = (size_t)py * job.W + px;
#pragma unroll
            for (int c = 0; c < DV; ++c) g[c] = job.dQ[p * DV + c];
            remaining = job.n_contrib[p];
        } else {
#pragma unroll
            for (int c = 0; c < DV; ++c) g[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int c = 0; c < DV; c += 2) {
            uint32_t h[4], l[4];
            const float4 a = g[c], b = c + 1 < DV ? g[c + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
            tc_split(a.x, a.y, h[0], l[0]);
            tc_split(a.z, a.w, h[1], l[1]);
            tc_split(b.x, b.y, h[2], l[2]);
            tc_split(b.z, b.w, h[3], l[3]);
            if (c + 1 < DV) {
                *reinterpret_cast<uint4*>(dq_hi + (size_t)t * DQS + 4 * c) = make_uint4(h[0], h[1], h[2], h[3]);
                *reinterpret_cast<uint4*>(dq_lo + (size_t)t * DQS + 4 * c) = make_uint4(l[0], l[1], l[2], l[3]);
            } else {
                *reinterpret_cast<uint2*>(dq_hi + (size_t)t * DQS + 4 * c) = make_uint2(h[0], h[1]);
                *reinterpret_cast<uint2*>(dq_lo + (size_t)t * DQS + 4 * c) = make_uint2(l[0], l[1]);
            }
        }
    }
    const int mt = warp & 3, nh = warp >> 2;  // GEMM role: Gaussian rows 16 mt.., channel half nh
    float T = 1.0f;
    bool done = remaining == 0;
    for (int start = range.x; start < range.y; start += kBwdBatch) {
        if (__syncthreads_count(done) == kTilePixels) break;
        const int cnt = min(kBwdBatch, range.y - start);
        if (t < cnt) {
            const int gid = job.pair_ids[start + t];
            s_xy[t] = job.xy[gid];
            s_co[t] = stage_splat(job.conic_opac[gid]);
            s_id[t] = gid;
        }
        __syncthreads();
        // 1. this pixel's weights for the batch (identical arithmetic to the forward pass); the
        //    columns of the Gaussians past the batch are zero
        for (int j = 0; j < kBwdBatch; ++j) {
            float w = 0.0f;
            if (j < cnt && !done) {
                const float alpha = splat_alpha(s_xy[j], s_co[j], fpx, fpy);
                if (alpha >= kAlphaMin) {
                    w = __fmul_rn(alpha, T);
                    T = __fmul_rn(T, __fsub_rn(1.0f, alpha));
                    if (--remaining == 0) done = true;
                }
            }
            const __nv_bfloat16 wh = __float2bfloat16_rn(w);
            wt_hi[(size_t)j * kWtStride + t] = wh;
            wt_lo[(size_t)j * kWtStride + t] = __float2bfloat16_rn(w - __bfloat162float(wh));
        }
        __syncthreads();
        // 2. warp (mt, nh): df rows 16 mt.. (Gaussians) x channels nh DQ/2.. over the 256 pixels
        if (16 * mt < cnt) {
            float acc[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
            const int ar = 16 * mt + (lane & 15), ac = (lane >> 4) * 8;  // A fragment row / column
            const int br = lane & 15;                                     // B fragment row (pixel)
#pragma unroll 4
            for (int kt = 0; kt < kTilePixels / 16; ++kt) {
                uint32_t ah[4], al[4];
                ldsm_x4(smem_addr(wt_hi + (size_t)ar * kWtStride + 16 * kt + ac), ah);
                ldsm_x4(smem_addr(wt_lo + (size_t)ar * kWtStride + 16 * kt + ac), al);
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const int col = nh * (DQ / 2) + 8 * n;
                    uint32_t bh[2], bl[2];
                    ldsm_x2_trans(smem_addr(dq_hi + (size_t)(16 * kt + br) * DQS + col), bh);
                    ldsm_x2_trans(smem_addr(dq_lo + (size_t)(16 * kt + br) * DQS + col), bl);
                    mma_bf16_16816(acc[n], ah, bh);
                    mma_bf16_16816(acc[n], ah, bl);
                    mma_bf16_16816(acc[n], al, bh);
                }
            }
            // 3. one atomic per non-zero (Gaussian, channel) of the tile
            const int g0 = 16 * mt + (lane >> 2);
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const int c = nh * (DQ / 2) + 8 * n + 2 * (lane & 3);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int g = g0 + 8 * h;
                    if (g >= cnt) continue;
                    float* dst = job.df + (size_t)s_id[g] * DQ + c;
                    if (acc[n][2 * h] != 0.0f) atomicAdd(dst, acc[n][2 * h]);
                    if (acc[n][2 * h + 1] != 0.0f) atomicAdd(dst + 1, acc[n][2 * h + 1]);
                }
            }
        }
        // the next batch's staging and W writes come after the barrier at the loop head
    }
}

template <int DQ>
__global__ void __launch_bounds__(kTilePixels) render_bwd_kernel(CamParams cam, const int2* __restrict__ ranges,
                                                                 const int32_t* __restrict__ pair_ids,
                                                                 const float2* __restrict__ xy,
                                                                 const float4* __restrict__ conic_opac,
                                                                 const int32_t* __restrict__ n_contrib,
                                                                 const float4* __restrict__ dQ, float* __restrict__ df) {
    extern __shared__ float4 smem_f4[];
    const int tile = cam.tile_order ? cam.tile_order[blockIdx.x] : (int)blockIdx.x;
    const TileJob job{tile, cam.tiles_x, cam.W, cam.H, ranges, pair_ids, xy, conic_opac, nullptr, nullptr, nullptr,
                      const_cast<int32_t*>(n_contrib), dQ, df};
    render_bwd_tile<DQ>(job, smem_f4);
}

// Persistent render backward over every tile of every frame of a batch, longest lists first
// (frames that share their queries add into the same df).
template <int DQ>
__global__ void __launch_bounds__(kTilePixels) render_bwd_batch_kernel(const __grid_constant__ BatchJobs jobs,
                                                                       const int32_t* __restrict__ order, int total,
                                                                       int* __restrict__ counter) {
    extern __shared__ float4 smem_f4[];
    for (int item = next_item(counter, order, total); item >= 0; item = next_item(counter, order, total)) {
        TileJob job = jobs.fr[item >> 20];
        job.tile = item & 0xFFFFF;
        render_bwd_tile<DQ>(job, smem_f4);
    }
}

// ---- the full Stage I render: queries, colours and depth blended together ---------------
//
// The colour c_i (view-independent) and the camera depth z_i of every Gaussian are blended with
// the same weights as its query (Eq. alpha_blending; the depth image uses the same blend).  The
// backward adds the gradients of the blend weights: with G = dL/dX the pixel's gradient over all
// blended channels X, and x_i the channels of contribution i,
//   dL/dalpha_i = T_i <G, x_i> - (<G, X> - P_i) / (1 - alpha_i),  P_i = sum_{k <= i} w_k <G, x_k>,
// so one running scalar per pixel replaces the back-to-front pass.  alpha = min(0.99, o e^power)
// passes dL/dalpha to o (e^power) and to power (alpha) unless it is clamped, and power to the
// screen mean and the conic.

template <int DQ>
__global__ void __launch_bounds__(fwd_threads<DQ>(), fwd_blocks<DQ>()) render_fwd_full_kernel(
    CamParams cam, const int2* __restrict__ ranges, const int32_t* __restrict__ pair_ids,
    const float2* __restrict__ xy, const float4* __restrict__ conic_opac, const float4* __restrict__ f,
    float4* __restrict__ Q, FullImages full, float* __restrict__ T_final, int32_t* __restrict__ n_contrib) {
    __shared__ FwdSmem<DQ, true> sm;
    const int tile = cam.tile_order ? cam.tile_order[blockIdx.x] : (int)blockIdx.x;
    const TileJob job{tile, cam.tiles_x, cam.W, cam.H, ranges, pair_ids, xy, conic_opac, f, Q, T_final, n_contrib,
                      nullptr, nullptr};
    render_fwd_tile<DQ, true>(job, sm, full);
}

// Backward of the full blend, a warp per strip of a tile and FP32 throughout (the geometry terms
// need <G, x_i>, a dot product over all channels, for every pixel and splat).  Per batch of 16
// Gaussians: (1) each lane takes its own pixels front to back from the strip's dQ rows in its
// registers: weight, <G, x_j>, dL/dalpha; the six geometry terms of its pixels are added over the
// warp by a reduce-scatter and leave with one atomic per term; the weights go to shared memory;
// (2) with lane = channel, the strip's dQ column in registers and the weights read as broadcasts,
// df_j[lane] = sum_p w_jp dQ_p[lane] leaves as one 128-byte atomic per Gaussian.  Reading the
// weights back instead of reducing 32 products over the warp takes 48 instructions where the 31
// shuffles with their selects took about 190.  Bound by issue.
// (640 x 480, 300k Gaussians, d = 32: 226 us with a block per tile and two warp reductions per
// Gaussian, 190-204 with the warp per strip.)
constexpr int kFullBatch = 16;
constexpr int kBwdWarps = 4;  // warps per block, each with strips of its own

template <int DQ>
constexpr int full_px() {  // pixels per lane (two at d = 32 take 220 registers: 8 warps per SM, 235 us
                            // against 190-204 at 640 x 480)
    return DQ <= 16 ? 2 : 1;
}

template <int DQ>
struct FullSmem {
    float w[kFullBatch][32 * full_px<DQ>() + 4];
    float4 f[kFullBatch][DQ / 4];
    float4 cz[kFullBatch];
    float4 co[kFullBatch];
    float2 xy[kFullBatch];
    int id[kFullBatch];
};

struct FullGrads {
    const float* Q;   // rendered images and their gradients
    const float* C;
    const float* Z;
    const float* dC;
    const float* dZ;
    float* dcol;      // N x 3
    float* dgeo;      // N x 8: d mean2d x, y, d conic a, b, c, d opacity, d depth channel, unused
};

template <int DQ>
__device__ __forceinline__ void render_bwd_full_strip(const TileJob& job, const FullImages& in, const FullGrads& out,
                                                      int strip, FullSmem<DQ>& sm) {
    constexpr int DV = DQ / 4, PX = full_px<DQ>(), SP = 32 * PX, ROWS = SP / kTile;
    constexpr int LC = DQ < 32 ? DQ : 32;       // channel lanes
    constexpr int CG = DQ > 32 ? DQ / 32 : 1;   // channels per lane
    constexpr int PC = SP * LC / 32;            // pixels of a lane's column
    const int tile = job.tile;
    const int tx = tile % job.tiles_x, ty = tile / job.tiles_x;
    const int lane = threadIdx.x & 31;
    const int x0 = tx * kTile, y0 = ty * kTile + strip * ROWS;
    const int px = x0 + (PX * lane) % kTile, py = y0 + PX * lane / kTile;
    const float fpy = (float)py;
    const int2 range = job.ranges[tile];
    int remaining[PX];
    int left = 0;
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        remaining[i] = px + i < job.W && py < job.H ? job.n_contrib[(size_t)py * job.W + px + i] : 0;
        left |= remaining[i];
    }
    if (range.x >= range.y || !__any_sync(0xffffffffu, left > 0)) return;
    // the lane's own rows G (queries, then colour and depth) and GX = <G, X>
    float4 g[PX][DV], gcz[PX];
    float GX[PX], P[PX], T[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        GX[i] = P[i] = 0.f;
        T[i] = 1.0f;
        gcz[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < DV; ++c) g[i][c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (px + i < job.W && py < job.H) {
            const size_t p = (size_t)py * job.W + px + i;
#pragma unroll
            for (int c = 0; c < DV; ++c) {
                const float4 v = job.dQ[p * DV + c], q = reinterpret_cast<const float4*>(out.Q)[p * DV + c];
                g[i][c] = v;
                GX[i] += v.x * q.x + v.y * q.y + v.z * q.z + v.w * q.w;
            }
            gcz[i] = make_float4(out.dC[3 * p], out.dC[3 * p + 1], out.dC[3 * p + 2], out.dZ[p]);
            GX[i] += gcz[i].x * out.C[3 * p] + gcz[i].y * out.C[3 * p + 1] + gcz[i].z * out.C[3 * p + 2] +
                     gcz[i].w * out.Z[p];
        }
    }
    // the lane's columns: channels lane % LC + 32 h of the strip's pixels (of half of them at
    // d = 16), and channel lane % 4 of colour and depth of SP / 8 of them
    const int first = PC * (lane / LC);
    float col[CG][PC], colz[SP / 8];
#pragma unroll
    for (int h = 0; h < CG; ++h)
#pragma unroll
        for (int k = 0; k < PC; ++k) {
            const int x = x0 + (first + k) % kTile, y = y0 + (first + k) / kTile;
            const float* d = reinterpret_cast<const float*>(job.dQ);
            col[h][k] = x < job.W && y < job.H ? d[((size_t)y * job.W + x) * DQ + 32 * h + lane % LC] : 0.f;
        }
#pragma unroll
    for (int k = 0; k < SP / 8; ++k) {
        const int i = (SP / 8) * (lane >> 2) + k, x = x0 + i % kTile, y = y0 + i / kTile;
        const size_t p = (size_t)y * job.W + x;
        colz[k] = x < job.W && y < job.H ? ((lane & 3) < 3 ? out.dC[3 * p + (lane & 3)] : out.dZ[p]) : 0.f;
    }
    for (int start = range.x; start < range.y; start += kFullBatch) {
        const int cnt = min(kFullBatch, range.y - start);
        __syncwarp();
        if (lane < cnt) {
            const int gid = job.pair_ids[start + lane];
            sm.id[lane] = gid;
            sm.xy[lane] = job.xy[gid];
            sm.co[lane] = stage_splat(job.conic_opac[gid]);
            sm.cz[lane] = make_float4(in.colours[3 * (size_t)gid], in.colours[3 * (size_t)gid + 1],
                                      in.colours[3 * (size_t)gid + 2], in.depth[gid]);
        }
        __syncwarp();
        for (int k = lane; k < cnt * DV; k += 32) sm.f[k / DV][k % DV] = job.f[(size_t)sm.id[k / DV] * DV + k % DV];
        __syncwarp();
        uint32_t hit = 0;  // Gaussians that reach the strip
        for (int j = 0; j < cnt; ++j) {
            const float2 m = sm.xy[j];
            const float4 q = sm.co[j];
            float w[PX], dx[PX], raw[PX], alpha[PX];
            const float dy = __fsub_rn(m.y, fpy);
            bool use[PX], any = false;
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                dx[i] = __fsub_rn(m.x, (float)(px + i));
                const float power = __fmaf_rn(dx[i], __fmaf_rn(q.x, dx[i], __fmul_rn(q.y, dy)),
                                              __fmul_rn(__fmul_rn(q.z, dy), dy));
                raw[i] = __fmul_rn(q.w, __expf(power));
                alpha[i] = fminf(kAlphaMax, raw[i]);
                use[i] = remaining[i] > 0 && power <= 0.0f && alpha[i] >= kAlphaMin;
                any = any || use[i];
            }
            if (!__any_sync(0xffffffffu, any)) continue;
            hit |= 1u << j;
            // <G, x_j>
            float gx[PX];
            {
                const float4 v = sm.cz[j];
#pragma unroll
                for (int i = 0; i < PX; ++i)
                    gx[i] = gcz[i].x * v.x + gcz[i].y * v.y + gcz[i].z * v.z + gcz[i].w * v.w;
            }
            Pair e[PX][2];  // two chains a pixel
#pragma unroll
            for (int i = 0; i < PX; ++i) e[i][0] = Pair(gx[i], 0.f), e[i][1] = Pair(0.f);
#pragma unroll
            for (int c = 0; c < DV; ++c) {
                const float4 v = sm.f[j][c];
#pragma unroll
                for (int i = 0; i < PX; ++i) {
                    e[i][0] = fma2(Pair(g[i][c].x, g[i][c].y), Pair(v.x, v.y), e[i][0]);
                    e[i][1] = fma2(Pair(g[i][c].z, g[i][c].w), Pair(v.z, v.w), e[i][1]);
                }
            }
            // d mean2d x, y, d conic a, b, c, d opacity of the lane's pixels
            float geo[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            const float ca = -2.0f * q.x, cb = -q.y, cc = -2.0f * q.z;
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                w[i] = 0.f;
                if (use[i]) {
                    float x, x1;
                    add2(e[i][0], e[i][1]).get(x, x1);
                    x += x1;
                    const float Tb = T[i];
                    w[i] = __fmul_rn(alpha[i], Tb);
                    T[i] = __fmul_rn(Tb, __fsub_rn(1.0f, alpha[i]));
                    --remaining[i];
                    P[i] += w[i] * x;
                    const float dalpha = Tb * x - (GX[i] - P[i]) / (1.0f - alpha[i]);
                    if (raw[i] <= kAlphaMax) {
                        const float dpow = dalpha * raw[i];
                        geo[0] += dpow * (-ca * dx[i] - cb * dy);
                        geo[1] += dpow * (-cb * dx[i] - cc * dy);
                        geo[2] += dpow * (-0.5f * dx[i] * dx[i]);
                        geo[3] += dpow * (-dx[i] * dy);
                        geo[4] += dpow * (-0.5f * dy * dy);
                        geo[5] += dalpha * (raw[i] / q.w);
                    }
                }
            }
            if (PX == 2)
                *reinterpret_cast<float2*>(&sm.w[j][2 * lane]) = make_float2(w[0], w[PX - 1]);
            else
                sm.w[j][lane] = w[0];
            // eight values (six used) scattered over lane bits 16, 8, 4, then added over 2 and 1
            const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float lo = geo[k], hi = k + 4 < 6 ? geo[k + 4 < 6 ? k + 4 : 0] : 0.f;
                const float r = __shfl_xor_sync(0xffffffffu, b4 ? lo : hi, 16);
                v[k] = (b4 ? hi : lo) + r;
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float r = __shfl_xor_sync(0xffffffffu, b3 ? v[k] : v[k + 2], 8);
                v[k] = (b3 ? v[k + 2] : v[k]) + r;
            }
            float s = (b2 ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, b2 ? v[0] : v[1], 4);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            const int slot = (b4 ? 4 : 0) + (b3 ? 2 : 0) + (b2 ? 1 : 0);
            if ((lane & 3) == 0 && slot < 6 && s != 0.0f) atomicAdd(out.dgeo + (size_t)sm.id[j] * 8 + slot, s);
        }
        __syncwarp();
        for (; hit; hit &= hit - 1) {
            const int j = __ffs(hit) - 1;
            const size_t gid = (size_t)sm.id[j];
            Pair a[CG][2];
#pragma unroll
            for (int h = 0; h < CG; ++h) a[h][0] = a[h][1] = Pair(0.f);
#pragma unroll
            for (int k = 0; k < PC; k += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sm.w[j][first + k]);
#pragma unroll
                for (int h = 0; h < CG; ++h) {
                    a[h][0] = fma2(Pair(v.x, v.y), Pair(col[h][k], col[h][k + 1]), a[h][0]);
                    a[h][1] = fma2(Pair(v.z, v.w), Pair(col[h][k + 2], col[h][k + 3]), a[h][1]);
                }
            }
            float az = 0.f;
#pragma unroll
            for (int k = 0; k < SP / 8; k += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sm.w[j][(SP / 8) * (lane >> 2) + k]);
                az += v.x * colz[k] + v.y * colz[k + 1] + v.z * colz[k + 2] + v.w * colz[k + 3];
            }
#pragma unroll
            for (int h = 0; h < CG; ++h) {
                float s, s1;
                add2(a[h][0], a[h][1]).get(s, s1);
                s += s1;
                if (LC == 16) s += __shfl_xor_sync(0xffffffffu, s, 16);
                if (lane < LC && s != 0.0f) atomicAdd(job.df + gid * DQ + 32 * h + lane, s);
            }
#pragma unroll
            for (int o = 16; o >= 4; o >>= 1) az += __shfl_xor_sync(0xffffffffu, az, o);
            if (lane < 4 && az != 0.0f) atomicAdd(lane < 3 ? out.dcol + gid * 3 + lane : out.dgeo + gid * 8 + 6, az);
        }
        left = 0;
#pragma unroll
        for (int i = 0; i < PX; ++i) left |= remaining[i];
        if (!__any_sync(0xffffffffu, left > 0)) break;
    }
}

template <int DQ>
__global__ void __launch_bounds__(32 * kBwdWarps, DQ == 32 ? 4 : 1) render_bwd_full_kernel(
    CamParams cam, const int2* __restrict__ ranges, const int32_t* __restrict__ pair_ids,
    const float2* __restrict__ xy, const float4* __restrict__ conic_opac, const float4* __restrict__ f, FullImages in,
    const int32_t* __restrict__ n_contrib, const float4* __restrict__ dQ, FullGrads out, float* __restrict__ df) {
    __shared__ __align__(16) FullSmem<DQ> sm[kBwdWarps];
    constexpr int strips = kTilePixels / (32 * full_px<DQ>());
    const int item = blockIdx.x * kBwdWarps + (threadIdx.x >> 5);
    const int t = item / strips;
    if (t >= cam.tiles_x * cam.tiles_y) return;
    const int tile = cam.tile_order ? cam.tile_order[t] : t;
    const TileJob job{tile, cam.tiles_x, cam.W, cam.H, ranges, pair_ids, xy, conic_opac, f, nullptr, nullptr,
                      const_cast<int32_t*>(n_contrib), dQ, df};
    render_bwd_full_strip<DQ>(job, in, out, item % strips, sm[threadIdx.x >> 5]);
}

template <int DQ>
latentam_status render_fwd_t(const CamParams& cam, const latentam_projected& proj, const latentam_bins& bins,
                             const float* f, float* Q, float* T_final, int32_t* n_contrib, cudaStream_t st) {
    const int tiles = cam.tiles_x * cam.tiles_y;
    render_fwd_kernel<DQ><<<tiles, fwd_threads<DQ>(), 0, st>>>(
        cam, reinterpret_cast<const int2*>(bins.tile_ranges), bins.pair_ids, reinterpret_cast<const float2*>(proj.xy),
        reinterpret_cast<const float4*>(proj.conic_opacity), reinterpret_cast<const float4*>(f),
        reinterpret_cast<float4*>(Q), T_final, n_contrib);
    LAT_CHECK_LAUNCH("render_fwd_kernel");
    return LATENTAM_OK;
}

// Dynamic shared memory of a kernel, set once per device.
template <auto Kern>
latentam_status bwd_smem(size_t smem) {
    static unsigned long long attr_set = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (!(attr_set & (1ull << (dev & 63)))) {
        cudaError_t e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_error(e, "render backward smem attribute");
        attr_set |= 1ull << (dev & 63);
    }
    return LATENTAM_OK;
}

template <int DQ>
latentam_status render_bwd_t(const CamParams& cam, const latentam_projected& proj, const latentam_bins& bins,
                             const int32_t* n_contrib, const float* dQ, float* df, int32_t n, cudaStream_t st,
                             bool accumulate) {
    if (!accumulate) {
        cudaError_t e = cudaMemsetAsync(df, 0, sizeof(float) * (size_t)n * DQ, st);
        if (e != cudaSuccess) return cuda_error(e, "memset df");
    }
    const int tiles = cam.tiles_x * cam.tiles_y;
    constexpr size_t smem = render_bwd_smem<DQ>();
    static_assert(smem <= 227 * 1024, "render backward tile does not fit in shared memory");
    LAT_TRY(bwd_smem<render_bwd_kernel<DQ>>(smem));
    render_bwd_kernel<DQ><<<tiles, kTilePixels, smem, st>>>(
        cam, reinterpret_cast<const int2*>(bins.tile_ranges), bins.pair_ids, reinterpret_cast<const float2*>(proj.xy),
        reinterpret_cast<const float4*>(proj.conic_opacity), n_contrib, reinterpret_cast<const float4*>(dQ), df);
    LAT_CHECK_LAUNCH("render_bwd_kernel");
    return LATENTAM_OK;
}

// Longest tiles first over every frame of a batch (the same length classes as
// a single frame's launch order); entries are (frame << 20) | tile.
__global__ void __launch_bounds__(1024) batch_order_kernel(const __grid_constant__ BatchJobs jobs,
                                                           int32_t* __restrict__ order) {
    __shared__ int s_cnt[33], s_pos[33];
    const int t = threadIdx.x;
    if (t < 33) s_cnt[t] = 0;
    __syncthreads();
    auto cls = [&](const TileJob& fr, int i) {
        const int2 r = fr.ranges[i];
        const int len = r.y - r.x;
        return len > 0 ? 32 - __clz(len) : 0;
    };
    for (int k = 0; k < jobs.n; ++k) {
        const TileJob& fr = jobs.fr[k];
        const int tiles = fr.tiles_x * ((fr.H + kTile - 1) / kTile);
        for (int i = t; i < tiles; i += blockDim.x) atomicAdd(&s_cnt[cls(fr, i)], 1);
    }
    __syncthreads();
    if (t == 0) {
        int run = 0;
        for (int c = 32; c >= 0; --c) {
            s_pos[c] = run;
            run += s_cnt[c];
        }
    }
    __syncthreads();
    for (int k = 0; k < jobs.n; ++k) {
        const TileJob& fr = jobs.fr[k];
        const int tiles = fr.tiles_x * ((fr.H + kTile - 1) / kTile);
        for (int i = t; i < tiles; i += blockDim.x) order[atomicAdd(&s_pos[cls(fr, i)], 1)] = (k << 20) | i;
    }
}

// CTAs of a persistent batch kernel: as many as can be resident at once, at most `total`.
template <auto Kern>
int persistent_grid(int threads, size_t smem, int total) {
    static int per_sm[64] = {0};  // of this kernel
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms = 1;
    int& b = per_sm[dev & 63];
    if (b == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, Kern, threads, smem) != cudaSuccess || b < 1) b = 1;
        (void)cudaGetLastError();
    }
    return std::max(1, std::min(total, b * sms));
}

template <int DQ>
latentam_status render_fwd_batch_t(const BatchJobs& jobs, const int32_t* order, int total, int* counter,
                                   cudaStream_t st) {
    constexpr int threads = fwd_threads<DQ>();
    render_fwd_batch_kernel<DQ><<<persistent_grid<render_fwd_batch_kernel<DQ>>(threads, 0, total), threads, 0, st>>>(
        jobs, order, total, counter);
    LAT_CHECK_LAUNCH("render_fwd_batch_kernel");
    return LATENTAM_OK;
}

template <int DQ>
latentam_status render_bwd_batch_t(const BatchJobs& jobs, const int32_t* order, int total, int* counter,
                                   cudaStream_t st) {
    constexpr size_t smem = render_bwd_smem<DQ>();
    LAT_TRY(bwd_smem<render_bwd_batch_kernel<DQ>>(smem));
    const int grid = persistent_grid<render_bwd_batch_kernel<DQ>>(kTilePixels, smem, total);
    render_bwd_batch_kernel<DQ><<<grid, kTilePixels, smem, st>>>(jobs, order, total, counter);
    LAT_CHECK_LAUNCH("render_bwd_batch_kernel");
    return LATENTAM_OK;
}

}  // namespace

latentam_status launch_batch_order(const BatchJobs& jobs, int32_t* order, cudaStream_t st) {
    batch_order_kernel<<<1, 1024, 0, st>>>(jobs, order);
    LAT_CHECK_LAUNCH("batch_order_kernel");
    return LATENTAM_OK;
}

latentam_status launch_render_fwd_batch(const BatchJobs& jobs, int d, const int32_t* order, int total, int* counter,
                                        cudaStream_t st) {
    if (total <= 0) return LATENTAM_OK;
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return cuda_error(e, "reset the render work ticket");
    switch (d) {
        case 16: return render_fwd_batch_t<16>(jobs, order, total, counter, st);
        case 32: return render_fwd_batch_t<32>(jobs, order, total, counter, st);
        case 64: return render_fwd_batch_t<64>(jobs, order, total, counter, st);
        default: set_error("query dimension d=%d not in {16, 32, 64}", d); return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
}

latentam_status launch_render_bwd_batch(const BatchJobs& jobs, int d, const int32_t* order, int total, int* counter,
                                        cudaStream_t st) {
    if (total <= 0) return LATENTAM_OK;
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return cuda_error(e, "reset the render work ticket");
    switch (d) {
        case 16: return render_bwd_batch_t<16>(jobs, order, total, counter, st);
        case 32: return render_bwd_batch_t<32>(jobs, order, total, counter, st);
        case 64: return render_bwd_batch_t<64>(jobs, order, total, counter, st);
        default: set_error("query dimension d=%d not in {16, 32, 64}", d); return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
}

latentam_status launch_render_fwd(const CamParams& cam, const latentam_projected& proj, const latentam_bins& bins,
                                  const float* f, int d, float* Q, float* T_final, int32_t* n_contrib,
                                  cudaStream_t st) {
    switch (d) {
        case 16: return render_fwd_t<16>(cam, proj, bins, f, Q, T_final, n_contrib, st);
        case 32: return render_fwd_t<32>(cam, proj, bins, f, Q, T_final, n_contrib, st);
        case 64: return render_fwd_t<64>(cam, proj, bins, f, Q, T_final, n_contrib, st);
        default: set_error("query dimension d=%d not in {16, 32, 64}", d); return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
}

latentam_status launch_render_full(const CamParams& cam, const latentam_projected& proj, const latentam_bins& bins,
                                   const float* f, int d, const float* colours, float* Q, float* C, float* Z,
                                   float* T_final, int32_t* n_contrib, cudaStream_t st) {
    const int tiles = cam.tiles_x * cam.tiles_y;
    auto args = [&](auto kernel, int threads) {
        kernel<<<tiles, threads, 0, st>>>(cam, reinterpret_cast<const int2*>(bins.tile_ranges), bins.pair_ids,
                                          reinterpret_cast<const float2*>(proj.xy),
                                          reinterpret_cast<const float4*>(proj.conic_opacity),
                                          reinterpret_cast<const float4*>(f), reinterpret_cast<float4*>(Q),
                                          FullImages{colours, proj.depth, C, Z}, T_final, n_contrib);
    };
    switch (d) {
        case 16: args(render_fwd_full_kernel<16>, fwd_threads<16>()); break;
        case 32: args(render_fwd_full_kernel<32>, fwd_threads<32>()); break;
        case 64: args(render_fwd_full_kernel<64>, fwd_threads<64>()); break;
        default: set_error("query dimension d=%d not in {16, 32, 64}", d); return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
    LAT_CHECK_LAUNCH("render_fwd_full_kernel");
    return LATENTAM_OK;
}

latentam_status launch_render_bwd_full(const CamParams& cam, const latentam_projected& proj,
                                       const latentam_bins& bins, const float* f, int d, const float* colours,
                                       const int32_t* n_contrib, const float* Q, const float* C, const float* Z,
                                       const float* dQ, const float* dC, const float* dZ, float* df, float* dcol,
                                       float* dgeo, int32_t n, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(df, 0, sizeof(float) * (size_t)n * d, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dcol, 0, sizeof(float) * (size_t)n * 3, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dgeo, 0, sizeof(float) * (size_t)n * 8, st);
    if (e != cudaSuccess) return cuda_error(e, "memset full gradients");
    const int tiles = cam.tiles_x * cam.tiles_y;
    auto args = [&](auto kernel, int strips) {
        kernel<<<(tiles * strips + kBwdWarps - 1) / kBwdWarps, 32 * kBwdWarps, 0, st>>>(
            cam, reinterpret_cast<const int2*>(bins.tile_ranges), bins.pair_ids, reinterpret_cast<const float2*>(proj.xy),
            reinterpret_cast<const float4*>(proj.conic_opacity), reinterpret_cast<const float4*>(f),
            FullImages{colours, proj.depth, nullptr, nullptr}, n_contrib, reinterpret_cast<const float4*>(dQ),
            FullGrads{Q, C, Z, dC, dZ, dcol, dgeo}, df);
    };
    switch (d) {
        case 16: args(render_bwd_full_kernel<16>, 8 / full_px<16>()); break;
        case 32: args(render_bwd_full_kernel<32>, 8 / full_px<32>()); break;
        case 64: args(render_bwd_full_kernel<64>, 8 / full_px<64>()); break;
        default: set_error("query dimension d=%d not in {16, 32, 64}", d); return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
    LAT_CHECK_LAUNCH("render_bwd_full_kernel");
    return LATENTAM_OK;
}

latentam_status launch_render_bwd(const CamParams& cam, const latentam_projected& proj, const latentam_bins& bins,
                                  const int32_t* n_contrib, const float* dQ, int d, float* df, int32_t n,
                                  cudaStream_t st, bool accumulate) {
    switch (d) {
        case 16: return render_bwd_t<16>(cam, proj, bins, n_contrib, dQ, df, n, st, accumulate);
        case 32: return render_bwd_t<32>(cam, proj, bins, n_contrib, dQ, df, n, st, accumulate);
        case 64: return render_bwd_t<64>(cam, proj, bins, n_contrib, dQ, df, n, st, accumulate);
        default: set_error("query dimension d=%d not in {16, 32, 64}", d); return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
}

}  // namespace lat

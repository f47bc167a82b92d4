// Query rendering Q = R_f(G, T) (Sec. III-B, Eq. render_query): the depth-ordered alpha
// blending of Eq. (alpha_blending) applied to the d-dimensional query vectors f_i, and its
// backward with respect to f.
//
// Forward: one CTA per 16x16 tile; the tile's Gaussians are staged through shared memory in
// batches (mean, exponent coefficients/opacity, query as float4 rows), so every query row is read
// from L2/HBM once per tile and broadcast to the 256 pixels.  Backward: one warp per 16x4 strip.
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
__global__ void __launch_bounds__(fwd_threads<DQ>(), 1) render_fwd_kernel(CamParams cam, const int2* __restrict__ ranges,
                                                                       const int32_t* __restrict__ pair_ids,
                                                                       const float2* __restrict__ xy,
                                                                       const float4* __restrict__ conic_opac,
                                                                       const float4* __restrict__ f,
                                                                       float4* __restrict__ Q,
                                                                       float* __restrict__ T_final,
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
__global__ void __launch_bounds__(fwd_threads<DQ>(), DQ == 32 ? 5 : 1) render_fwd_batch_kernel(const __grid_constant__ BatchJobs jobs,
                                                                             const int32_t* __restrict__ order,
                                                                             int total, int* __restrict__ counter) {
    __shared__ FwdSmem<DQ> sm;
    for (int item = next_item(counter, order, total); item >= 0; item = next_item(counter, order, total)) {
        TileJob job = jobs.fr[item >> 20];
        job.tile = item & 0xFFFFF;
        render_fwd_tile<DQ>(job, sm);
    }
}

// Backward of the query blend, df_i = sum_p w_ip dQ_p, as one small GEMM per strip (16 x 4 pixels) and
// batch of 32 Gaussians on the tensor cores, a warp to itself: each lane recomputes the weights of
// two horizontally adjacent pixels front to back (the forward's arithmetic, so the same
// contributions are taken: a pixel stops after its n_contrib-th one) into the warp's shared-memory
// matrix W^T (Gaussians x pixels), each weight as two BF16 terms w = hi + lo (hi = bf16(w),
// lo = bf16(w - hi)); the strip's dQ rows are held the same way, for d <= 32 as B fragments in
// registers for the whole list.  mma.sync m16n8k16 (BF16 in, FP32 accumulate) then sums
// W_hi dQ_hi + W_hi dQ_lo + W_lo dQ_hi over the 64 pixels (each product within 2^-16 of the FP32
// one), and lane pairs trade halves so that the non-zero sums go to df as 16-byte atomics.
// Bound by issue and latency of the weight chains: warps share nothing, so there are no block
// barriers, each strip stops at its own last contribution, and 10 KB of shared memory per warp
// leaves the registers to limit the warps in flight.  (A block per tile with a 256 x 64 weight
// matrix and the tile's dQ in shared memory held two blocks per SM and three barriers a batch.)
// A per-strip contraction of 32 x 64 x d does not amortise TMEM allocation and completion waits;
// the warp-level MMA runs in the registers of the warp that computed the weights.
// (848 x 480, 200k Gaussians, d = 32: 74 us with the block per tile, 48 with the warp per strip.)
constexpr int kBwdBatch = 32;
constexpr int kStripRows = 4;
constexpr int kStrips = kTile / kStripRows;       // strips per tile
constexpr int kStripPixels = kTile * kStripRows;  // 64: two per lane
constexpr int kWtStride = kStripPixels + 8;       // bf16 per W^T row (144 B: ldmatrix rows on distinct banks)

template <int DQ>
struct BwdSmem {
    __nv_bfloat16 w[2][kBwdBatch][kWtStride];  // W^T hi, lo
    // dQ hi, lo; for d <= 32 one plane at a time passes through w on its way to the registers
    __nv_bfloat16 dq[DQ <= 32 ? 1 : 2][DQ <= 32 ? 1 : kStripPixels][DQ + 8];
    float4 co[kBwdBatch];
    float2 xy[kBwdBatch];
    int id[kBwdBatch];
    __device__ __forceinline__ __nv_bfloat16* dq_row(int plane, int pixel) {
        return DQ <= 32 ? &w[0][0][0] + pixel * (DQ + 8) : &dq[DQ <= 32 ? 0 : plane][DQ <= 32 ? 0 : pixel][0];
    }
};
static_assert(sizeof(__nv_bfloat16) * kStripPixels * (32 + 8) <= sizeof(BwdSmem<32>::w), "a dQ plane fits in w");
static_assert(sizeof(BwdSmem<16>) % 16 == 0 && sizeof(BwdSmem<32>) % 16 == 0 && sizeof(BwdSmem<64>) % 16 == 0,
              "16-byte rows");

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

// The m16n8 accumulator tile (rows = Gaussians r0 .. r0 + 15 of the batch, columns = channels
// c0 .. c0 + 7) added to dst rows of `ld` floats: an even lane ends with four consecutive channels of
// its upper row, an odd lane of its lower row.  vec: dst and ld are multiples of 16 bytes.
__device__ __forceinline__ void add_tile(const float (&c)[4], const int* id, int r0, int rows, int c0, float* dst,
                                         int ld, bool vec, int lane) {
    const bool odd = lane & 1;
    const float s0 = odd ? c[0] : c[2], s1 = odd ? c[1] : c[3];
    const float o0 = __shfl_xor_sync(0xffffffffu, s0, 1), o1 = __shfl_xor_sync(0xffffffffu, s1, 1);
    const float4 v = odd ? make_float4(o0, o1, c[2], c[3]) : make_float4(c[0], c[1], o0, o1);
    const int r = r0 + (lane >> 2) + (odd ? 8 : 0);
    if (r >= rows) return;
    float* p = dst + (size_t)id[r] * ld + c0 + 4 * ((lane & 3) >> 1);
    if (vec) {
        if (v.x != 0.0f || v.y != 0.0f || v.z != 0.0f || v.w != 0.0f) atomicAdd(reinterpret_cast<float4*>(p), v);
    } else {
        if (v.x != 0.0f) atomicAdd(p, v.x);
        if (v.y != 0.0f) atomicAdd(p + 1, v.y);
        if (v.z != 0.0f) atomicAdd(p + 2, v.z);
        if (v.w != 0.0f) atomicAdd(p + 3, v.w);
    }
}

// Backward of one strip by one warp.
template <int DQ>
__device__ __forceinline__ void render_bwd_strip(const TileJob& job, int strip, BwdSmem<DQ>& sm) {
    constexpr int DV = DQ / 4, NT = DQ / 8, KT = kStripPixels / 16;
    constexpr bool REG = DQ <= 32;  // dQ fragments in registers
    const int tile = job.tile;
    const int tx = tile % job.tiles_x, ty = tile / job.tiles_x;
    const int lane = threadIdx.x & 31;
    const int px = tx * kTile + (2 * lane) % kTile, py = ty * kTile + strip * kStripRows + lane / (kTile / 2);
    const float fpx[2] = {(float)px, (float)(px + 1)}, fpy = (float)py;
    const int2 range = job.ranges[tile];
    const bool vec = (reinterpret_cast<uintptr_t>(job.df) & 15u) == 0;
    int remaining[2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
        remaining[i] = px + i < job.W && py < job.H ? job.n_contrib[(size_t)py * job.W + px + i] : 0;
    if (range.x >= range.y || !__any_sync(0xffffffffu, (remaining[0] | remaining[1]) > 0)) return;
    // the strip's dQ rows (pixel 2 lane + i) as hi / lo terms
    uint32_t bh[REG ? KT : 1][REG ? NT : 1][2], bl[REG ? KT : 1][REG ? NT : 1][2];
    {
        uint32_t lo[2][DQ / 2];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const bool in = px + i < job.W && py < job.H;
            const size_t p = (size_t)py * job.W + px + i;
#pragma unroll
            for (int c = 0; c < DV; ++c) {
                const float4 g = in ? job.dQ[p * DV + c] : make_float4(0.f, 0.f, 0.f, 0.f);
                uint32_t h0, h1;
                tc_split(g.x, g.y, h0, lo[i][2 * c]);
                tc_split(g.z, g.w, h1, lo[i][2 * c + 1]);
                *reinterpret_cast<uint2*>(sm.dq_row(0, 2 * lane + i) + 4 * c) = make_uint2(h0, h1);
            }
        }
        auto put_lo = [&](int plane) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int c = 0; c < DV; ++c)
                    *reinterpret_cast<uint2*>(sm.dq_row(plane, 2 * lane + i) + 4 * c) =
                        make_uint2(lo[i][2 * c], lo[i][2 * c + 1]);
        };
        auto fragments = [&](uint32_t (&b)[REG ? KT : 1][REG ? NT : 1][2]) {
#pragma unroll
            for (int kt = 0; kt < (REG ? KT : 0); ++kt)
#pragma unroll
                for (int n = 0; n < NT; ++n)
                    ldsm_x2_trans(smem_addr(sm.dq_row(0, 16 * kt + (lane & 15)) + 8 * n), b[kt][n]);
        };
        if (REG) {
            __syncwarp();
            fragments(bh);
            __syncwarp();
            put_lo(0);
            __syncwarp();
            fragments(bl);
        } else {
            put_lo(1);
        }
    }
    float T[2] = {1.0f, 1.0f};
    // the splats of the next batch are fetched while this one is worked on
    int gid = 0;
    float2 nxy = make_float2(0.f, 0.f);
    float4 nco = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int start) {
        if (start + lane < range.y) {
            gid = job.pair_ids[start + lane];
            nxy = job.xy[gid];
            nco = job.conic_opac[gid];
        }
    };
    fetch(range.x);
    for (int start = range.x; start < range.y; start += kBwdBatch) {
        const int cnt = min(kBwdBatch, range.y - start);
        __syncwarp();
        sm.xy[lane] = nxy;
        sm.co[lane] = stage_splat(nco);
        sm.id[lane] = gid;
        __syncwarp();
        fetch(start + kBwdBatch);
        // 1. the lane's weights for the batch (identical arithmetic to the forward pass)
#pragma unroll 2
        for (int j = 0; j < cnt; ++j) {
            const float2 m = sm.xy[j];
            const float4 q = sm.co[j];
            float w[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float alpha = splat_alpha(m, q, fpx[i], fpy);
                const bool use = remaining[i] > 0 && alpha >= kAlphaMin;
                w[i] = use ? __fmul_rn(alpha, T[i]) : 0.0f;
                if (use) {
                    T[i] = __fmul_rn(T[i], __fsub_rn(1.0f, alpha));
                    --remaining[i];
                }
            }
            uint32_t h, l;
            tc_split(w[0], w[1], h, l);
            *reinterpret_cast<uint32_t*>(&sm.w[0][j][2 * lane]) = h;
            *reinterpret_cast<uint32_t*>(&sm.w[1][j][2 * lane]) = l;
        }
        __syncwarp();
        // 2. df rows (16 Gaussians) x channels over the strip's 64 pixels; rows past the batch hold
        //    leftovers and are not added
        for (int r0 = 0; r0 < cnt; r0 += 16) {
            float acc[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
#pragma unroll
            for (int kt = 0; kt < KT; ++kt) {
                uint32_t ah[4], al[4];
                ldsm_x4(smem_addr(&sm.w[0][r0 + (lane & 15)][16 * kt + (lane >> 4) * 8]), ah);
                ldsm_x4(smem_addr(&sm.w[1][r0 + (lane & 15)][16 * kt + (lane >> 4) * 8]), al);
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    uint32_t fh[2], fl[2];
                    if (REG) {
                        fh[0] = bh[REG ? kt : 0][REG ? n : 0][0], fh[1] = bh[REG ? kt : 0][REG ? n : 0][1];
                        fl[0] = bl[REG ? kt : 0][REG ? n : 0][0], fl[1] = bl[REG ? kt : 0][REG ? n : 0][1];
                    } else {
                        ldsm_x2_trans(smem_addr(sm.dq_row(0, 16 * kt + (lane & 15)) + 8 * n), fh);
                        ldsm_x2_trans(smem_addr(sm.dq_row(1, 16 * kt + (lane & 15)) + 8 * n), fl);
                    }
                    mma_bf16_16816(acc[n], ah, fh);
                    mma_bf16_16816(acc[n], ah, fl);
                    mma_bf16_16816(acc[n], al, fh);
                }
            }
            // 3. the non-zero sums of the strip
#pragma unroll
            for (int n = 0; n < NT; ++n) add_tile(acc[n], sm.id, r0, cnt, 8 * n, job.df, DQ, vec, lane);
        }
        if (!__any_sync(0xffffffffu, (remaining[0] | remaining[1]) > 0)) break;
    }
}

constexpr int kBwdWarps = 4;  // warps per block, each with strips of its own

template <int DQ>
__global__ void __launch_bounds__(32 * kBwdWarps) render_bwd_kernel(CamParams cam, const int2* __restrict__ ranges,
                                                                    const int32_t* __restrict__ pair_ids,
                                                                    const float2* __restrict__ xy,
                                                                    const float4* __restrict__ conic_opac,
                                                                    const int32_t* __restrict__ n_contrib,
                                                                    const float4* __restrict__ dQ,
                                                                    float* __restrict__ df) {
    extern __shared__ float4 smem_f4[];
    const int item = blockIdx.x * kBwdWarps + (threadIdx.x >> 5);
    const int t = item / kStrips;
    if (t >= cam.tiles_x * cam.tiles_y) return;
    const int tile = cam.tile_order ? cam.tile_order[t] : t;
    const TileJob job{tile, cam.tiles_x, cam.W, cam.H, ranges, pair_ids, xy, conic_opac, nullptr, nullptr, nullptr,
                      const_cast<int32_t*>(n_contrib), dQ, df};
    render_bwd_strip<DQ>(job, item % kStrips, reinterpret_cast<BwdSmem<DQ>*>(smem_f4)[threadIdx.x >> 5]);
}

// Persistent render backward over every strip of every tile of a batch, longest lists first, each
// warp with a ticket of its own (frames that share their queries add into the same df).
template <int DQ>
__global__ void __launch_bounds__(32 * kBwdWarps) render_bwd_batch_kernel(const __grid_constant__ BatchJobs jobs,
                                                                          const int32_t* __restrict__ order,
                                                                          int total, int* __restrict__ counter) {
    extern __shared__ float4 smem_f4[];
    BwdSmem<DQ>& sm = reinterpret_cast<BwdSmem<DQ>*>(smem_f4)[threadIdx.x >> 5];
    for (;;) {
        int it = 0;
        if ((threadIdx.x & 31) == 0) it = atomicAdd(counter, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= total * kStrips) return;
        const int item = order[it / kStrips];
        TileJob job = jobs.fr[item >> 20];
        job.tile = item & 0xFFFFF;
        render_bwd_strip<DQ>(job, it % kStrips, sm);
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
__global__ void __launch_bounds__(fwd_threads<DQ>(), 1) render_fwd_full_kernel(
    CamParams cam, const int2* __restrict__ ranges, const int32_t* __restrict__ pair_ids,
    const float2* __restrict__ xy, const float4* __restrict__ conic_opac, const float4* __restrict__ f,
    float4* __restrict__ Q, FullImages full, float* __restrict__ T_final, int32_t* __restrict__ n_contrib) {
    __shared__ FwdSmem<DQ, true> sm;
    const int tile = cam.tile_order ? cam.tile_order[blockIdx.x] : (int)blockIdx.x;
    const TileJob job{tile, cam.tiles_x, cam.W, cam.H, ranges, pair_ids, xy, conic_opac, f, Q, T_final, n_contrib,
                      nullptr, nullptr};
    render_fwd_tile<DQ, true>(job, sm, full);
}

// Backward of the full blend, a warp per strip as above but in FP32 throughout (the geometry terms
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
    constexpr size_t smem = sizeof(BwdSmem<DQ>) * kBwdWarps;
    LAT_TRY(bwd_smem<render_bwd_kernel<DQ>>(smem));
    render_bwd_kernel<DQ><<<(tiles * kStrips + kBwdWarps - 1) / kBwdWarps, 32 * kBwdWarps, smem, st>>>(
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
    constexpr size_t smem = sizeof(BwdSmem<DQ>) * kBwdWarps;
    constexpr int threads = 32 * kBwdWarps;
    LAT_TRY(bwd_smem<render_bwd_batch_kernel<DQ>>(smem));
    const int grid = persistent_grid<render_bwd_batch_kernel<DQ>>(threads, smem, total);
    render_bwd_batch_kernel<DQ><<<grid, threads, smem, st>>>(jobs, order, total, counter);
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

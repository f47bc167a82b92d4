// Streaming K-means update of the dictionary atoms (Algorithm 1, Eq. stream_kmeans_init,
// Sec. III-C): the new keyframe's embeddings are summarised into k micro-clusters by a local
// K-means, which are merged with the weighted global centres and re-clustered to the fixed
// dictionary size K.  Global centres keep their slots (row j stays row j); weight 0 marks an
// empty slot, and the empty slots take the heaviest micro-centres first.
//
// Local phase (n rows, k <= 32 centres): one pass over the rows per Lloyd iteration.  A warp
// holds four rows in registers (eight up to D = 256), finds each one's nearest centre against the
// centres staged in shared memory (squared distance as |c|^2 - 2 <x, c>, ties to the lower index)
// and adds the rows to its own copy of the cluster sums in shared memory; copies and blocks are
// summed in a fixed order (no atomics), so the result does not depend on scheduling.
// Global phase (at most K + k weighted points against K centres): an FP32 tiled product of the
// points with the centres whose epilogue keeps each point's nearest occupied slot as one 64-bit
// atomic minimum of (distance, slot), then one block per centre gathers its points' weighted sum
// in point order.
#include <algorithm>

#include "internal.cuh"

namespace lat {
namespace {

constexpr int kMaxMicro = 32;
constexpr int kRowWarps = 8;                // warps per block of the local pass, at most
constexpr size_t kRowSmem = 220 * 1024;     // shared memory one block of it may take
constexpr int kAccumThreads = 256;

__device__ __forceinline__ float warp_allsum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// |x|^2 of a row, every lane (lane l takes x[l], x[l + 32], ... in order).
__device__ __forceinline__ float warp_norm2(const float* x, int D, int lane) {
    float s = 0.f;
    for (int j = lane; j < D; j += 32) s += x[j] * x[j];
    return warp_allsum(s);
}

// ---- local phase ------------------------------------------------------------------------

// C[c] = F[init_idx[c]]; an index outside [0, n) starts its centre at the origin.
__global__ void local_init(const float* __restrict__ F, int64_t n, int D, const int32_t* __restrict__ init_idx,
                           float* __restrict__ C) {
    const int c = blockIdx.x;
    const int32_t r = init_idx[c];
    const bool ok = r >= 0 && (int64_t)r < n;
    for (int j = threadIdx.x; j < D; j += blockDim.x) C[(int64_t)c * D + j] = ok ? F[(int64_t)r * D + j] : 0.f;
}

// Launch shape of the local pass.  Row warps per block (a power of two: eight, fewer when there are
// fewer rows than that many warps take), the copies of the k x D sums they share (a power of two; 0
// when k x D is too large for even one beside the staged centres), rows per warp and blocks.
struct PassShape {
    int warps, copies, rows, per_sm, nb;
    size_t smem;
};

// Two blocks per SM up to D = 512 (64 registers of embeddings a lane at four rows of 512), one
// above (128 registers), so that 128 KB of rows per SM are in flight either way; of the shapes
// that fit, the one with the most copies.
PassShape pass_shape(int64_t n, int k, int D, int sms) {
    PassShape p{};
    p.rows = D <= 256 ? 8 : 4;
    const int64_t groups = (n + p.rows - 1) / p.rows;
    p.warps = 1;
    while (p.warps < kRowWarps && (int64_t)p.warps * sms < groups) p.warps *= 2;
    auto bytes = [&](int copies) { return sizeof(float) * ((size_t)(copies + 1) * k * D + k); };
    for (p.per_sm = D <= 512 ? 2 : 1; p.per_sm >= 1 && !p.copies; --p.per_sm)
        for (p.copies = p.warps; p.copies && bytes(p.copies) > kRowSmem / p.per_sm; p.copies /= 2) {
        }
    ++p.per_sm;
    p.smem = bytes(p.copies);
    p.nb = (int)std::max<int64_t>(1, std::min<int64_t>((groups + p.warps - 1) / p.warps, (int64_t)p.per_sm * sms));
    return p;
}

__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// One Lloyd pass: every valid row's nearest centre and the block's sums of its rows per cluster,
// part[block] (k x D) and pcnt[block] (k).  Bound by the read of the embeddings (HBM, once per
// iteration; the earlier assign / accumulate pair read them twice and held one row per warp).
// R rows per warp: each centre quad read from shared memory meets 4 R products, and the R dot
// products leave the butterfly together (log2 R scatter steps, then the R lane groups each finish
// one row), in the summation tree of a plain butterfly.  Rows of one group that share their
// cluster are added together before the read-modify-write of the sums.  NV: quads per lane
// (D <= 128 NV).  `warps` of the block's eight take rows, all of them stage the centres and add up
// the copies.  With fewer copies of the sums than row warps, the warps of a copy add in turn, round
// by round (warp w hands over to w + copies, the last one to the first one's next round), each
// handover a named barrier of the two warps; every row warp runs every round.
// At 307,200 x 512, k = 5: 252 + 185 us (assign, accumulate) -> 126 us, 5.0 TB/s.
template <int NV, int R>
__global__ void __launch_bounds__(32 * kRowWarps, NV <= 4 ? 2 : 1) local_pass(const float* __restrict__ F, int64_t n, int D,
                                                                const uint8_t* __restrict__ valid,
                                                                const float* __restrict__ C, int k,
                                                                int warps, int copies,
                                                                int32_t* __restrict__ assign,
                                                                float* __restrict__ part, int32_t* __restrict__ pcnt) {
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_cnt[kRowWarps][kMaxMicro];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int D4 = D / 4;
    float4* sC = reinterpret_cast<float4*>(sm);        // k x D
    float4* sS = sC + (size_t)k * D4;                  // copies x k x D
    float* sN = sm + (size_t)(copies + 1) * k * D;     // k
    for (int i = threadIdx.x; i < k * D4; i += blockDim.x) sC[i] = reinterpret_cast<const float4*>(C)[i];
    for (int i = threadIdx.x; i < copies * k * D4; i += blockDim.x) sS[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int c = warp; c < k; c += kRowWarps) {
        const float s = warp_norm2(sm + (size_t)c * D, D, lane);
        if (lane == 0) sN[c] = s;
    }
    __syncthreads();
    // lane l only touches quads l, l + 32, ... of its warp's copy
    float4* own = sS + (size_t)(warp % copies) * k * D4;
    const bool turns = copies < warps, last = warp + copies >= warps;
    int cnt = 0;                               // rows of cluster `lane`
    constexpr int G = 32 / R;                  // lanes that end with one row's dot product
    const float4* F4 = reinterpret_cast<const float4*>(F);
    const int64_t step = (int64_t)gridDim.x * warps * R, begin = (int64_t)blockIdx.x * warps * R;
    const int64_t rounds = warp < warps && begin < n ? (n - begin + step - 1) / step : 0;  // the same for all row warps
    for (int64_t round = 0; round < rounds; ++round) {
        const int64_t r0 = begin + round * step + warp * R;
        float4 x[R][NV];
        bool ok[R];
#pragma unroll
        for (int r = 0; r < R; ++r) ok[r] = r0 + r < n && (!valid || valid[r0 + r]);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int q = lane + 32 * i;
                x[r][i] = ok[r] && q < D4 ? __ldcs(F4 + (r0 + r) * D4 + q) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        float best = INFINITY;
        int bi = 0;
        for (int c = 0; c < k; ++c) {
            float s[R];
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = 0.f;
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int q = lane + 32 * i;
                if (q < D4) {
                    const float4 cc = sC[c * D4 + q];
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        s[r] += x[r][i].x * cc.x + x[r][i].y * cc.y + x[r][i].z * cc.z + x[r][i].w * cc.w;
                }
            }
#pragma unroll
            for (int half = R / 2, o = 16; half >= 1; half >>= 1, o >>= 1) {
                const bool upper = (lane & o) != 0;
#pragma unroll
                for (int r = 0; r < half; ++r) {
                    const float send = upper ? s[r] : s[r + half], keep = upper ? s[r + half] : s[r];
                    s[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
#pragma unroll
            for (int o = G / 2; o >= 1; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
            const float v = sN[c] - 2.0f * s[0];
            if (v < best) best = v, bi = c;
        }
        int a[R];
        bool same = true;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            a[r] = __shfl_sync(0xffffffffu, bi, G * r);
            if (!ok[r]) a[r] = -1;
            same = same && a[r] == a[0];
            cnt += a[r] == lane ? 1 : 0;
            if (assign && lane == 0 && r0 + r < n) assign[r0 + r] = a[r];
        }
        auto add = [&](int c, const float4 (&y)[NV]) {
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int q = lane + 32 * i;
                if (q < D4) {
                    float4 t = own[c * D4 + q];
                    t.x += y[i].x, t.y += y[i].y, t.z += y[i].z, t.w += y[i].w;
                    own[c * D4 + q] = t;
                }
            }
        };
        __syncwarp();  // named barriers are for whole warps
        if (turns && (warp >= copies || round > 0)) pair_sync(1 + warp);
        if (same) {
            if (a[0] >= 0) {
#pragma unroll
                for (int r = 1; r < R; ++r)
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        x[0][i].x += x[r][i].x, x[0][i].y += x[r][i].y;
                        x[0][i].z += x[r][i].z, x[0][i].w += x[r][i].w;
                    }
                add(a[0], x[0]);
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (a[r] >= 0) add(a[r], x[r]);
        }
        __syncwarp();
        if (turns && !(last && round + 1 == rounds)) pair_arrive(last ? 1 + warp % copies : 1 + warp + copies);
    }
    s_cnt[warp][lane] = cnt;
    __syncthreads();
    for (int i = threadIdx.x; i < k * D4; i += blockDim.x) {
        float4 t = sS[i];
        for (int w = 1; w < copies; ++w) {
            const float4 u = sS[(size_t)w * k * D4 + i];
            t.x += u.x, t.y += u.y, t.z += u.z, t.w += u.w;
        }
        reinterpret_cast<float4*>(part + (size_t)blockIdx.x * k * D)[i] = t;
    }
    if (threadIdx.x < k) {
        int t = 0;
        for (int w = 0; w < warps; ++w) t += s_cnt[w][threadIdx.x];
        pcnt[(size_t)blockIdx.x * k + threadIdx.x] = t;
    }
}

// assign[r] = nearest of the k centres (-1 for an invalid row); warp per row.  Shared memory:
// the centres (k x D) and their squared norms.  D % 4 == 0, D <= 1024.  With local_accum, the
// form for k x D past what local_pass holds twice in shared memory (k = 32 at D > 876).
__global__ void __launch_bounds__(256) local_assign(const float* __restrict__ F, int64_t n, int D,
                                                    const uint8_t* __restrict__ valid, const float* __restrict__ C,
                                                    int k, int32_t* __restrict__ assign) {
    extern __shared__ __align__(16) float sm[];
    float* sC = sm;
    float* sN = sm + (size_t)k * D;
    const int D4 = D / 4;
    const float4* C4 = reinterpret_cast<const float4*>(C);
    float4* sC4 = reinterpret_cast<float4*>(sC);
    for (int i = threadIdx.x; i < k * D4; i += blockDim.x) sC4[i] = C4[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c = warp; c < k; c += 8) {
        const float s = warp_norm2(sC + (size_t)c * D, D, lane);
        if (lane == 0) sN[c] = s;
    }
    __syncthreads();
    const float4* F4 = reinterpret_cast<const float4*>(F);
    for (int64_t r = (int64_t)blockIdx.x * 8 + warp; r < n; r += (int64_t)gridDim.x * 8) {
        if (valid && !valid[r]) {
            if (lane == 0) assign[r] = -1;
            continue;
        }
        float4 x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int q = lane + 32 * i;
            x[i] = q < D4 ? F4[r * D4 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        float best = INFINITY;
        int bi = 0;
        for (int c = 0; c < k; ++c) {
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int q = lane + 32 * i;
                if (q < D4) {
                    const float4 cc = sC4[(size_t)c * D4 + q];
                    s += x[i].x * cc.x + x[i].y * cc.y + x[i].z * cc.z + x[i].w * cc.w;
                }
            }
            s = warp_allsum(s);
            const float v = sN[c] - 2.0f * s;
            if (v < best) {
                best = v;
                bi = c;
            }
        }
        if (lane == 0) assign[r] = bi;
    }
}

// Per-block cluster sums of rows [b R, (b+1) R): G = 256 / (D/4) row groups, each with its
// own accumulator copy (k x D) in shared memory; thread t of group g owns columns
// 4 (t mod D/4) .. +3 and adds rows g, g+G, ... of the range in order.  The copies are added in
// group order into part[b] (k x D); pcnt[b] (k) counts the rows.
__global__ void __launch_bounds__(kAccumThreads) local_accum(const float* __restrict__ F, int64_t n, int D,
                                                             const int32_t* __restrict__ assign, int k, int64_t R,
                                                             float* __restrict__ part, int32_t* __restrict__ pcnt) {
    extern __shared__ __align__(16) float acc[];  // G x k x D
    __shared__ int cnt[kMaxMicro];
    const int D4 = D / 4;
    const int G = kAccumThreads / D4;  // row groups; threads past G * D4 (D4 not dividing 256) idle
    const int t = threadIdx.x, g = t / D4, q = t % D4;
    for (int i = t; i < G * k * D; i += kAccumThreads) acc[i] = 0.f;
    if (t < k) cnt[t] = 0;
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * R, r1 = min(n, r0 + R);
    const float4* F4 = reinterpret_cast<const float4*>(F);
    float4* a4 = reinterpret_cast<float4*>(acc) + (size_t)min(g, G - 1) * k * D4;
    constexpr int U = 4;
    for (int64_t rb = r0 + g; g < G && rb < r1; rb += (int64_t)G * U) {
        int cs[U];
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t r = rb + (int64_t)u * G;
            cs[u] = r < r1 ? assign[r] : -1;
            v[u] = cs[u] >= 0 ? F4[r * D4 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (cs[u] < 0) continue;
            float4& s = a4[(size_t)cs[u] * D4 + q];
            s.x += v[u].x, s.y += v[u].y, s.z += v[u].z, s.w += v[u].w;
        }
    }
    __syncthreads();
    if (t == 0) {  // row counts, in row order
        for (int64_t r = r0; r < r1; ++r) {
            const int c = assign[r];
            if (c >= 0) ++cnt[c];
        }
    }
    __syncthreads();
    for (int i = t; i < k * D; i += kAccumThreads) {
        float s = 0.f;
        for (int h = 0; h < G; ++h) s += acc[(size_t)h * k * D + i];
        part[(int64_t)blockIdx.x * k * D + i] = s;
    }
    if (t < k) pcnt[(int64_t)blockIdx.x * k + t] = cnt[t];
}

// C[c][j] = (sum over blocks of part[b][c][j]) / count_c, kept when the cluster is empty;
// W[c] = count_c.  Block per 32 columns of the k x D sums, warp w takes blocks w, w + 32, ... and the
// warps' sums are added in order.  (One thread per column walking all blocks took 43 us over 304
// blocks at k = 5, D = 512.)
constexpr int kFinishWarps = 32;
__global__ void __launch_bounds__(32 * kFinishWarps) local_finish(const float* __restrict__ part,
                                                                  const int32_t* __restrict__ pcnt, int nb, int k,
                                                                  int D, float* __restrict__ C,
                                                                  float* __restrict__ W) {
    __shared__ float s_sum[kFinishWarps][32];
    __shared__ long long s_cnt[kFinishWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane, kD = k * D;
    const int c = min(i, kD - 1) / D;
    float s = 0.f;
    long long m = 0;
    if (i < kD) {
#pragma unroll 4
        for (int b = warp; b < nb; b += kFinishWarps) {
            s += part[(size_t)b * kD + i];
            m += pcnt[(size_t)b * k + c];
        }
    }
    s_sum[warp][lane] = s;
    s_cnt[warp][lane] = m;
    __syncthreads();
    if (warp != 0 || i >= kD) return;
#pragma unroll
    for (int w = 1; w < kFinishWarps; ++w) s += s_sum[w][lane], m += s_cnt[w][lane];
    if (m > 0) C[i] = s / (float)m;
    if (i == c * D) W[c] = (float)m;
}

// ---- global phase -----------------------------------------------------------------------

struct MergeBufs {
    int32_t* n_points;   // [0] = |P|
    int32_t* pt_src;     // K + k: slot j >= 0, or micro c as -1 - c
    float* pt_w;         // K + k
    int32_t* slot_fill;  // K: micro index copied into an empty slot, or -1
    int32_t* active;     // K: 1 = the slot competes in the re-clustering
};

// One block of 1024 threads: the point list, the fill of the empty slots and the active set.
__global__ void __launch_bounds__(1024) global_merge(const float* __restrict__ w, int K, const float* __restrict__ mW,
                                                     int k, MergeBufs b) {
    __shared__ int by_rank[kMaxMicro];
    __shared__ int live_before[kMaxMicro + 1];
    __shared__ int warp_tot[2][32];
    __shared__ int carry[2];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) {
        int lv = 0;
        for (int c = 0; c < k; ++c) {
            live_before[c] = lv;
            lv += mW[c] > 0.f ? 1 : 0;
        }
        live_before[k] = lv;
        carry[0] = carry[1] = 0;
    }
    if (t < k && mW[t] > 0.f) {  // rank among the live micro-centres: heavier first, then lower index
        int r = 0;
        for (int c = 0; c < k; ++c)
            if (mW[c] > 0.f && (mW[c] > mW[t] || (mW[c] == mW[t] && c < t))) ++r;
        by_rank[r] = t;
    }
    __syncthreads();
    const int n_live = live_before[k];
    for (int base = 0; base < K; base += 1024) {
        const int j = base + t;
        const int used = (j < K && w[j] > 0.f) ? 1 : 0;
        const int empty = (j < K && !used) ? 1 : 0;
        int xu = used, xe = empty;
        for (int o = 1; o < 32; o <<= 1) {
            const int yu = __shfl_up_sync(0xffffffffu, xu, o), ye = __shfl_up_sync(0xffffffffu, xe, o);
            if (lane >= o) xu += yu, xe += ye;
        }
        if (lane == 31) warp_tot[0][warp] = xu, warp_tot[1][warp] = xe;
        __syncthreads();
        if (warp == 0) {
            int wu = warp_tot[0][lane], we = warp_tot[1][lane];
            for (int o = 1; o < 32; o <<= 1) {
                const int yu = __shfl_up_sync(0xffffffffu, wu, o), ye = __shfl_up_sync(0xffffffffu, we, o);
                if (lane >= o) wu += yu, we += ye;
            }
            warp_tot[0][lane] = wu, warp_tot[1][lane] = we;
        }
        __syncthreads();
        const int ub = carry[0] + (warp ? warp_tot[0][warp - 1] : 0) + xu - used;
        const int eb = carry[1] + (warp ? warp_tot[1][warp - 1] : 0) + xe - empty;
        if (j < K) {
            b.slot_fill[j] = -1;
            if (used) {
                b.pt_src[ub] = j;
                b.pt_w[ub] = w[j];
                b.active[j] = 1;
            } else if (eb < n_live) {
                b.slot_fill[j] = by_rank[eb];
                b.active[j] = 1;
            } else {
                b.active[j] = 0;
            }
        }
        __syncthreads();
        if (t == 1023) carry[0] = ub + used, carry[1] = eb + empty;
        __syncthreads();
    }
    const int U = carry[0];
    if (t < k && mW[t] > 0.f) {
        b.pt_src[U + live_before[t]] = -1 - t;
        b.pt_w[U + live_before[t]] = mW[t];
    }
    if (t == 0) b.n_points[0] = U + n_live;
}

// Rows and keys of the re-clustering.  Block b: point b (an occupied slot of C, or a micro-centre;
// zero past the last one) into Pm, its assignment and keys cleared; slot b: an empty slot that takes
// a micro-centre starts there, and the slot's squared norm.
__global__ void __launch_bounds__(256) global_setup(float* __restrict__ C, const float* __restrict__ mC, int K, int KP,
                                                    int D, MergeBufs b, float* __restrict__ Pm,
                                                    float* __restrict__ nrm, uint64_t* __restrict__ keys,
                                                    int32_t* __restrict__ pa) {
    const int i = blockIdx.x, t = threadIdx.x;
    if (i < KP) {
        const int s = i < b.n_points[0] ? b.pt_src[i] : 0;
        const bool live = i < b.n_points[0];
        const float* src = s >= 0 ? C + (int64_t)s * D : mC + (int64_t)(-1 - s) * D;
        for (int j = t; j < D; j += 256) Pm[(int64_t)i * D + j] = live ? src[j] : 0.f;
        if (t == 0) {
            keys[i] = keys[KP + i] = ~0ull;
            if (pa) pa[i] = -1;
        }
    }
    if (i < K) {
        const int c = b.slot_fill[i];
        const float* src = c >= 0 ? mC + (int64_t)c * D : C + (int64_t)i * D;
        if (c >= 0)
            for (int j = t; j < D; j += 256) C[(int64_t)i * D + j] = src[j];
        if (t < 32) {
            const float s = warp_norm2(src, D, t);
            if (t == 0) nrm[i] = s;
        }
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool in) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int bytes = in ? 16 : 0;  // the rest is zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// (distance, slot) as one word whose unsigned order is distance first, then the lower slot.
__device__ __forceinline__ uint64_t nearest_key(float v, int c) {
    uint32_t u = __float_as_uint(v + 0.0f);  // -0 and +0 are the same distance
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((uint64_t)u << 32) | (uint32_t)c;
}

// keys[p] = minimum over the active slots c of (nrm[c] - 2 <Pm_p, C_c>, c): TP x TC tiles of the
// points' products with the slots, FP32 FMAs with D in order, operands by cp.async through a ring
// of `kDistStages` slices of BK; each thread MP x MC products (rows a half-warp apart).  A distance
// that is not below infinity takes no slot.
constexpr int kDistStages = 4;

template <int TP, int TC, int BK>
constexpr size_t dist_smem() {
    return sizeof(float) * kDistStages * (size_t)(TP + TC) * (BK + 4);
}

template <int TP, int TC, int THREADS, int BK>
__global__ void __launch_bounds__(THREADS) global_nearest(const float* __restrict__ Pm, int KP,
                                                          const float* __restrict__ C, int K, int D, MergeBufs b,
                                                          const float* __restrict__ nrm,
                                                          unsigned long long* __restrict__ keys) {
    constexpr int LD = BK + 4;  // padded rows: eight rows of 16 bytes cover the banks once
    constexpr int MP = TP / (THREADS / 16), MC = TC / 16;
    extern __shared__ __align__(16) float sm[];
    const int P = b.n_points[0];
    const int p0 = blockIdx.y * TP, c0 = blockIdx.x * TC;
    const int t = threadIdx.x, tc = t & 15, tp = t >> 4;
    // nothing to do past the last point, or where every slot of the tile is empty
    if (p0 >= P || !__syncthreads_or(t < TC && c0 + t < K && b.active[c0 + t])) return;
    const int slices = (D + BK - 1) / BK;
    auto load = [&](int s) {
        float* dst = sm + (size_t)(s % kDistStages) * (TP + TC) * LD;
        for (int i = t; i < (TP + TC) * (BK / 4); i += THREADS) {
            const int row = i / (BK / 4), col = s * BK + 4 * (i % (BK / 4));
            const bool point = row < TP;
            const int g = point ? p0 + row : c0 + row - TP;
            const bool in = col < D && g < (point ? KP : K);
            const float* src = (point ? Pm : C) + (in ? (int64_t)g * D + col : 0);
            cp_async16(dst + row * LD + 4 * (i % (BK / 4)), src, in);
        }
    };
    float acc[MP][MC];
#pragma unroll
    for (int i = 0; i < MP; ++i)
#pragma unroll
        for (int j = 0; j < MC; ++j) acc[i][j] = 0.f;
#pragma unroll
    for (int s = 0; s < kDistStages - 1; ++s) {
        if (s < slices) load(s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int s = 0; s < slices; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kDistStages - 2) : "memory");
        __syncthreads();
        if (s + kDistStages - 1 < slices) load(s + kDistStages - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* A = sm + (size_t)(s % kDistStages) * (TP + TC) * LD;
        const float* B = A + TP * LD;
#pragma unroll 4
        for (int kk = 0; kk < BK; kk += 4) {
            float4 a[MP], c[MC];
#pragma unroll
            for (int i = 0; i < MP; ++i)
                a[i] = *reinterpret_cast<const float4*>(A + (tp + (THREADS / 16) * i) * LD + kk);
#pragma unroll
            for (int j = 0; j < MC; ++j) c[j] = *reinterpret_cast<const float4*>(B + (tc + 16 * j) * LD + kk);
#pragma unroll
            for (int i = 0; i < MP; ++i)
#pragma unroll
                for (int j = 0; j < MC; ++j) {
                    float v = acc[i][j];
                    v = fmaf(a[i].x, c[j].x, v);
                    v = fmaf(a[i].y, c[j].y, v);
                    v = fmaf(a[i].z, c[j].z, v);
                    acc[i][j] = fmaf(a[i].w, c[j].w, v);
                }
        }
    }
#pragma unroll
    for (int i = 0; i < MP; ++i) {
        const int p = p0 + tp + (THREADS / 16) * i;
        uint64_t key = ~0ull;
#pragma unroll
        for (int j = 0; j < MC; ++j) {
            const int c = c0 + tc + 16 * j;
            if (c < K && b.active[c]) {
                const float v = nrm[c] - 2.0f * acc[i][j];
                if (v < INFINITY) key = min(key, nearest_key(v, c));
            }
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) key = min(key, (uint64_t)__shfl_xor_sync(0xffffffffu, key, o));
        if (tc == 0 && p < P && key != ~0ull) atomicMin(keys + p, (unsigned long long)key);
    }
}

// Block per slot: the weighted mean of its points (in point order), their total weight and the
// new row's squared norm; an active slot without points keeps its position with weight 0; inactive
// slots are left.  The points' keys are read 256 at a time and the slot's own compacted in order.
// `next` (the other half of the keys) is cleared for the next iteration; pa (nullable): every
// point's slot.
__global__ void __launch_bounds__(256) global_update(const float* __restrict__ Pm, int K, int KP, int D, MergeBufs b,
                                                     const uint64_t* __restrict__ keys, uint64_t* __restrict__ next,
                                                     int32_t* __restrict__ pa, float* __restrict__ C,
                                                     float* __restrict__ W, float* __restrict__ nrm) {
    __shared__ int s_p[256], s_n[8];
    __shared__ float s_w[256];
    __shared__ float s_row[1024];
    const int c = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int P = b.n_points[0];
    for (int p = c * 256 + t; p < KP; p += K * 256) next[p] = ~0ull;
    if (pa)
        for (int p = c * 256 + t; p < P; p += K * 256) pa[p] = keys[p] == ~0ull ? 0x7fffffff : (int32_t)(uint32_t)keys[p];
    if (!b.active[c]) return;
    constexpr int kCols = 4;  // D <= 1024 = 4 x 256
    float acc[kCols] = {0.f, 0.f, 0.f, 0.f};
    float wsum = 0.f;
    for (int base = 0; base < P; base += 256) {
        const int p = base + t;
        const bool mine = p < P && (uint32_t)keys[p] == (uint32_t)c;
        const uint32_t vote = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) s_n[warp] = __popc(vote);
        __syncthreads();
        int at = __popc(vote & ((1u << lane) - 1u)), members = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += s_n[w];
            members += s_n[w];
        }
        if (mine) s_p[at] = p, s_w[at] = b.pt_w[p];
        __syncthreads();
#pragma unroll 4
        for (int m = 0; m < members; ++m) {
            const float wp = s_w[m];
            const float* row = Pm + (int64_t)s_p[m] * D;
            wsum += wp;
#pragma unroll
            for (int u = 0; u < kCols; ++u) {
                const int j = t + 256 * u;
                if (j < D) acc[u] += wp * row[j];
            }
        }
        __syncthreads();
    }
    if (t == 0) W[c] = wsum;
    if (!(wsum > 0.f)) return;
#pragma unroll
    for (int u = 0; u < kCols; ++u) {
        const int j = t + 256 * u;
        if (j < D) {
            const float v = acc[u] / wsum;
            C[(int64_t)c * D + j] = v;
            s_row[j] = v;
        }
    }
    __syncthreads();
    if (warp == 0) {
        const float s = warp_norm2(s_row, D, lane);
        if (lane == 0) nrm[c] = s;
    }
}

template <int TP, int TC, int THREADS, int BK>
latentam_status launch_nearest(const float* Pm, int KP, const float* C, int K, int D, const MergeBufs& mb,
                               const float* nrm, uint64_t* keys, cudaStream_t st) {
    constexpr size_t smem = dist_smem<TP, TC, BK>();
    auto kern = global_nearest<TP, TC, THREADS, BK>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(e, "kmeans global_nearest smem attribute");
    kern<<<dim3((K + TC - 1) / TC, (KP + TP - 1) / TP), THREADS, smem, st>>>(
        Pm, KP, C, K, D, mb, nrm, reinterpret_cast<unsigned long long*>(keys));
    LAT_CHECK_LAUNCH("kmeans global_nearest");
    return LATENTAM_OK;
}

template <int NV, int R>
latentam_status launch_pass(const KMeansArgs& a, const float* C, const PassShape& p, int32_t* assign, float* part,
                            int32_t* pcnt, cudaStream_t st) {
    auto kern = local_pass<NV, R>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return cuda_error(e, "kmeans local_pass smem attribute");
    kern<<<p.nb, 32 * kRowWarps, p.smem, st>>>(a.F, a.n, a.D, a.valid, C, a.k, p.warps, p.copies, assign, part, pcnt);
    LAT_CHECK_LAUNCH("kmeans local_pass");
    return LATENTAM_OK;
}

latentam_status pass(const KMeansArgs& a, const float* C, const PassShape& p, int32_t* assign, float* part,
                     int32_t* pcnt, cudaStream_t st) {
    switch ((a.D + 127) / 128) {
        case 1: return launch_pass<1, 8>(a, C, p, assign, part, pcnt, st);
        case 2: return launch_pass<2, 8>(a, C, p, assign, part, pcnt, st);
        case 3: return launch_pass<3, 4>(a, C, p, assign, part, pcnt, st);
        case 4: return launch_pass<4, 4>(a, C, p, assign, part, pcnt, st);
        case 5:
        case 6: return launch_pass<6, 4>(a, C, p, assign, part, pcnt, st);
        default: return launch_pass<8, 4>(a, C, p, assign, part, pcnt, st);
    }
}

}  // namespace

latentam_status stream_kmeans(latentam_ctx* ctx, const KMeansArgs& a, cudaStream_t st) {
    const int k = a.k, K = a.K, D = a.D, KP = K + k;
    const int64_t n = a.n;
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const int sms = ctx->num_sms;
    const PassShape shape = pass_shape(n, k, D, sms);
    const bool fused = shape.copies > 0;
    const int nb = fused ? shape.nb : (int)std::min<int64_t>((n + 63) / 64, 2 * (int64_t)sms);
    const size_t part_b = up(4 * (size_t)nb * k * D), pcnt_b = up(4 * (size_t)nb * k);
    const size_t asg_b = fused || a.micro_assign ? 0 : up(4 * (size_t)std::max<int64_t>(n, 1));
    const size_t bytes = (a.micro_C ? 0 : up(4 * (size_t)k * D)) + (a.micro_W ? 0 : up(4 * (size_t)k)) + up(4) +
                         2 * up(4 * (size_t)KP) + up(16 * (size_t)KP) + 3 * up(4 * (size_t)K) +
                         up(4 * (size_t)KP * D) + part_b + pcnt_b + asg_b;
    char* base = static_cast<char*>(ws(ctx, WS_KMEANS, bytes));
    if (!base) return LATENTAM_ERR_OUT_OF_MEMORY;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        char* p = base + o;
        o += up(bytes);
        return p;
    };
    // the buffers whose sizes do not depend on n first: their addresses (and the global
    // phase's captured graph) then stay the same from one keyframe to the next
    float* mC = a.micro_C ? a.micro_C : reinterpret_cast<float*>(take(4 * (size_t)k * D));
    float* mW = a.micro_W ? a.micro_W : reinterpret_cast<float*>(take(4 * (size_t)k));
    MergeBufs mb;
    mb.n_points = reinterpret_cast<int32_t*>(take(4));
    mb.pt_src = reinterpret_cast<int32_t*>(take(4 * (size_t)KP));
    mb.pt_w = reinterpret_cast<float*>(take(4 * (size_t)KP));
    uint64_t* keys = reinterpret_cast<uint64_t*>(take(16 * (size_t)KP));  // two halves, used in turn
    mb.slot_fill = reinterpret_cast<int32_t*>(take(4 * (size_t)K));
    mb.active = reinterpret_cast<int32_t*>(take(4 * (size_t)K));
    float* nrm = reinterpret_cast<float*>(take(4 * (size_t)K));
    float* Pm = reinterpret_cast<float*>(take(4 * (size_t)KP * D));
    float* part = reinterpret_cast<float*>(take(part_b));
    int32_t* pcnt = reinterpret_cast<int32_t*>(take(pcnt_b));
    int32_t* asg = a.micro_assign || fused ? a.micro_assign : reinterpret_cast<int32_t*>(take(asg_b));

    // Both phases are chains of small dependent launches with no host round trip: each replays
    // a captured CUDA graph once the same shapes and buffers recur (the global phase's shapes
    // are the dictionary's, the same for every keyframe; the local phase's depend on the
    // number of targets).
    auto local = [&](cudaStream_t s) -> latentam_status {
        local_init<<<k, 256, 0, s>>>(a.F, n, D, a.init_idx, mC);
        LAT_CHECK_LAUNCH("kmeans local_init");
        for (int it = 0; it < a.iters_local; ++it) {
            if (fused) {
                LAT_TRY(pass(a, mC, shape, it + 1 == a.iters_local ? asg : nullptr, part, pcnt, s));
            } else {
                const size_t sm_assign = 4 * ((size_t)k * D + k);
                const size_t sm_accum = 4 * (size_t)(kAccumThreads / (D / 4)) * k * D;
                const int ga = (int)std::max<int64_t>(1, std::min<int64_t>((n + 7) / 8, 4 * (int64_t)sms));
                cudaFuncSetAttribute(local_assign, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_assign);
                cudaFuncSetAttribute(local_accum, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_accum);
                local_assign<<<ga, 256, sm_assign, s>>>(a.F, n, D, a.valid, mC, k, asg);
                LAT_CHECK_LAUNCH("kmeans local_assign");
                local_accum<<<nb, kAccumThreads, sm_accum, s>>>(a.F, n, D, asg, k, (n + nb - 1) / nb, part, pcnt);
                LAT_CHECK_LAUNCH("kmeans local_accum");
            }
            local_finish<<<(k * D + 31) / 32, 32 * kFinishWarps, 0, s>>>(part, pcnt, nb, k, D, mC, mW);
            LAT_CHECK_LAUNCH("kmeans local_finish");
        }
        return LATENTAM_OK;
    };
    auto global = [&](cudaStream_t s) -> latentam_status {
        global_merge<<<1, 1024, 0, s>>>(a.weights, K, mW, k, mb);
        LAT_CHECK_LAUNCH("kmeans global_merge");
        global_setup<<<KP, 256, 0, s>>>(a.centres, mC, K, KP, D, mb, Pm, nrm, keys, a.point_assign);
        LAT_CHECK_LAUNCH("kmeans global_setup");
        const int64_t small_tiles = (int64_t)((KP + 15) / 16) * ((K + 31) / 32);
        for (int it = 0; it < a.iters_global; ++it) {
            uint64_t *cur = keys + (it & 1 ? KP : 0), *next = keys + (it & 1 ? 0 : KP);
            // 16 x 32 tiles while all of them are resident at once (four blocks per SM), else 64 x 64
            if (small_tiles <= 4 * sms)
                LAT_TRY((launch_nearest<16, 32, 256, 64>(Pm, KP, a.centres, K, D, mb, nrm, cur, s)));
            else
                LAT_TRY((launch_nearest<64, 64, 256, 32>(Pm, KP, a.centres, K, D, mb, nrm, cur, s)));
            global_update<<<K, 256, 0, s>>>(Pm, K, KP, D, mb, cur, next,
                                            it + 1 == a.iters_global ? a.point_assign : nullptr, a.centres, a.weights,
                                            nrm);
            LAT_CHECK_LAUNCH("kmeans global_update");
        }
        return LATENTAM_OK;
    };
    const uint64_t lkey[] = {0x6b6d2d6c6f63616cull /* tag: local phase */, (uint64_t)n, (uint64_t)D, (uint64_t)k,
                             (uint64_t)a.iters_local, reinterpret_cast<uint64_t>(a.F),
                             reinterpret_cast<uint64_t>(a.valid), reinterpret_cast<uint64_t>(a.init_idx),
                             reinterpret_cast<uint64_t>(mC), reinterpret_cast<uint64_t>(mW),
                             reinterpret_cast<uint64_t>(asg), reinterpret_cast<uint64_t>(part),
                             reinterpret_cast<uint64_t>(st), ctx->ws_generation};
    LAT_TRY(cached_launch(ctx, lkey, (int)(sizeof(lkey) / sizeof(lkey[0])), st, local));
    const uint64_t gkey[] = {0x6b6d2d676c6f6262ull /* tag: global phase */, (uint64_t)D, (uint64_t)k, (uint64_t)K,
                             (uint64_t)a.iters_global, reinterpret_cast<uint64_t>(a.centres),
                             reinterpret_cast<uint64_t>(a.weights), reinterpret_cast<uint64_t>(mC),
                             reinterpret_cast<uint64_t>(mW), reinterpret_cast<uint64_t>(a.point_assign),
                             reinterpret_cast<uint64_t>(base), reinterpret_cast<uint64_t>(st), ctx->ws_generation};
    LAT_TRY(cached_launch(ctx, gkey, (int)(sizeof(gkey) / sizeof(gkey[0])), st, global));
    return LATENTAM_OK;
}

}  // namespace lat

// Tile binning and sorting of the splats (the depth-ordered lists that Eq. alpha_blending
// walks, Sec. III-A):
//   1. the number of splats of every tile (one atomic per covered tile)
//   2. per-tile [start, end) ranges and the pair count P: one scan of the tiles in a single launch
//      (decoupled look-back across blocks, a bounded wait)
//   3. each pair's Gaussian into its tile's range, in the order of the atomics, and the tiles' launch
//      order (longest lists first)
//   4. each tile's list sorted by (binary32 depth key, index) in shared memory, which makes the
//      lists an exact function of the splats whatever order they arrived in
// The host reads P once, while step 3 runs: the launches after step 2 need only the buffers'
// capacity, and do nothing when P exceeds it.  Bound by launches and by the dependent loads of
// each small kernel.  (An exclusive scan of tiles-touched, emission in index order and a stable
// radix sort of the pairs on the tile bits took 14 launches and the host read between them:
// 62 us of kernels for 85,000 pairs of 300,000 Gaussians in 1,200 tiles; these four take 31.)
#include <algorithm>

#include "internal.cuh"

namespace lat {
namespace {

constexpr int kScanTiles = 64;            // tiles per block of tile_scan, one per thread
constexpr int kBinThreads = 256;
constexpr int64_t kMaxPairs = (1ll << 30) - 1;
constexpr int kSpinLimit = 1 << 20;
constexpr int kTestSpinLimit = 1 << 12;   // the short limit of an armed test stall

// Look-back words of tile_scan: per block its own pair count, flagged as an aggregate, later
// replaced by the inclusive count of every block up to and including it.
constexpr uint64_t kLbAggregate = 1ull << 62;
constexpr uint64_t kLbInclusive = 2ull << 62;
constexpr uint64_t kLbValue = kLbAggregate - 1ull;

__device__ __forceinline__ uint64_t ld_relaxed_gpu(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_gpu(uint64_t* p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The counters of one binning, in one zeroed block of memory (see bin_words): per tile the splats
// counted and the splats placed, kTileWords apart (packed, the atomics of a few hundred tiles meet in
// a few L2 lines: 610,000 pairs in 300 tiles 103 us to count and 91 to place, 40 and 42 at 8 words, 17
// and 21 at a line of 32), the look-back words (one more, never written: what an armed test stall
// polls), the block ticket.
constexpr int kTileWords = 32;
struct BinWords {
    uint64_t* status;
    uint32_t *count, *placed, *ticket;
};

size_t bin_words_bytes(int64_t tiles) {
    const int64_t nb = (tiles + kScanTiles - 1) / kScanTiles;
    return 8 * (size_t)(nb + 1) + 4 * (size_t)(kTileWords * tiles + 1);
}

BinWords bin_words(void* base, int64_t tiles) {
    const int64_t nb = (tiles + kScanTiles - 1) / kScanTiles;
    BinWords w;
    w.status = static_cast<uint64_t*>(base);
    w.count = reinterpret_cast<uint32_t*>(w.status + nb + 1);
    w.placed = w.count + 1;
    w.ticket = w.count + kTileWords * tiles;
    return w;
}

// Warps that share the pairs of 32 splats (a power of two): one where the splats alone give every SM
// eight warps, up to 64 where a few splats may cover the image (5 splats of 22,500 pairs: 156 us to
// count and 438 to place with one warp, the whole binning 545 -> 40).
int pair_parts(int N, int sms) {
    const int64_t groups = ((int64_t)N + 31) / 32;
    int parts = 1;
    while (parts < 64 && groups * parts * 2 <= 8 * (int64_t)sms) parts *= 2;
    return parts;
}

// body(g, tile) for every pair of 32 consecutive splats, of those of warp `index` (of the grid; parts
// warps to 32 splats), 32 pairs at a time: each lane finds its pair's splat in the prefix sums of the
// counts, so that a splat of many tiles does not leave 31 lanes waiting and the pairs' atomics
// overlap.  A splat's pairs are its first tiles_touched tiles in row order, those of the image.  For
// full warps.
template <class Body>
__device__ __forceinline__ void warp_pairs(int index, int parts, int N, const int32_t* __restrict__ touched,
                                           const int4* __restrict__ rect, int tiles_x, int tiles, Body&& body) {
    const int lane = threadIdx.x & 31, part = index & (parts - 1);
    const int64_t first = (int64_t)(index / parts) * 32;
    if (first >= N) return;
    const int g = (int)first + lane;
    int n = g < N ? touched[g] : 0;
    int x0 = 0, y0 = 0, w = 1;
    if (n > 0) {
        const int4 r = rect[g];
        x0 = r.x, y0 = r.y, w = max(r.z - r.x, 0);
        n = min(n, w * max(r.w - r.y, 0));
    }
    n = max(n, 0);
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    const int all = __shfl_sync(0xffffffffu, incl, 31), before = incl - n;
    for (int i0 = 32 * part; i0 < all; i0 += 32 * parts) {
        const int i = i0 + lane;
        int own = 0;  // splats of the warp whose pairs all come before pair i
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, incl, own + o - 1) <= i) own += o;
        own = min(own, 31);
        const int k = i - __shfl_sync(0xffffffffu, before, own), ow = __shfl_sync(0xffffffffu, w, own);
        const int ox = __shfl_sync(0xffffffffu, x0, own), oy = __shfl_sync(0xffffffffu, y0, own);
        if (i < all) {
            const int row = k / ow, t = (oy + row) * tiles_x + ox + k - row * ow;
            if (t >= 0 && t < tiles) body(g - lane + own, t);
        }
    }
}

// Also hands the slot's error words of earlier calls to the host (err: a look-back that gave up;
// tc_flag: a tensor-core kernel's wait).
__global__ void __launch_bounds__(kBinThreads) count_tiles(int N, int parts, const int32_t* __restrict__ touched,
                                                           const int4* __restrict__ rect, int tiles_x, int tiles,
                                                           uint32_t* __restrict__ count, const uint32_t* err,
                                                           const int* tc_flag, volatile uint32_t* host) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        host[2] = *err;
        host[3] = (uint32_t)*tc_flag;
    }
    warp_pairs((int)(blockIdx.x * (kBinThreads / 32) + threadIdx.x / 32), parts, N, touched, rect, tiles_x, tiles,
               [&](int, int t) { atomicAdd(count + (size_t)t * kTileWords, 1u); });
}

// Ranges of 64 consecutive tiles per block, the blocks in ticket order (so that every block before
// one belongs to a block already running), each adding the pairs of the earlier blocks: one warp
// reads 32 of their words at a time until it meets an inclusive one.  The waits are bounded
// (spin_limit polls): a walk that gives up raises *err, so that the later steps leave every tile
// empty, and adds up the earlier tiles' counts itself, so that the pair count stays exact.
// stall_block >= 0 (a test of that path) makes that block's first look-back poll the word that
// nothing writes, so that its wait runs out.
__global__ void __launch_bounds__(kScanTiles) tile_scan(BinWords w, int tiles, int2* __restrict__ ranges,
                                                        uint32_t* __restrict__ total, volatile uint32_t* host,
                                                        uint32_t* err, int spin_limit, int stall_block) {
    __shared__ uint32_t s_block, s_half;
    __shared__ uint64_t s_earlier;
    const int t = threadIdx.x, lane = t & 31, nb = gridDim.x;
    if (t == 0) s_block = atomicAdd(w.ticket, 1u);
    __syncthreads();
    const int b = (int)s_block, tile = b * kScanTiles + t;
    const uint32_t c = tile < tiles ? w.count[(size_t)tile * kTileWords] : 0u;
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (t == 31) s_half = incl;
    __syncthreads();
    if (t >= 32) incl += s_half;
    if (t == kScanTiles - 1) {
        s_earlier = 0;
        st_relaxed_gpu(w.status + b, (b == 0 ? kLbInclusive : kLbAggregate) | incl);
    }
    __syncthreads();
    if (b > 0 && t < 32) {
        uint64_t sum = 0;
        bool ok = true;
        for (int last = b - 1; last >= 0 && ok; last -= 32) {
            const int j = last - lane;
            const uint64_t* word = b == stall_block && j == b - 1 ? w.status + nb : w.status + j;
            uint64_t v = 0;
            int spins = 0;
            while (true) {
                if (j >= 0 && v == 0) v = ld_relaxed_gpu(word);
                if (__all_sync(0xffffffffu, j < 0 || v != 0)) break;
                if (++spins >= spin_limit) {
                    ok = false;
                    break;
                }
                if (spins >= 32) __nanosleep(64);
            }
            const uint32_t full = __ballot_sync(0xffffffffu, (v & kLbInclusive) != 0);
            const int stop = full ? __ffs(full) - 1 : 31;  // the nearest inclusive word counts last
            uint64_t x = lane <= stop ? v & kLbValue : 0ull;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            sum += x;
            if (full) break;
        }
        if (!ok) {
            sum = 0;
            for (int i = lane; i < b * kScanTiles; i += 32) sum += w.count[(size_t)i * kTileWords];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
        if (lane == 0) {
            if (!ok) atomicExch(err, 1u);
            s_earlier = sum;
        }
    }
    __syncthreads();
    const uint64_t end = s_earlier + incl;
    if (tile < tiles) ranges[tile] = make_int2((int)(end - c), (int)end);
    if (t == kScanTiles - 1) {
        if (b > 0) st_relaxed_gpu(w.status + b, kLbInclusive | end);
        if (b == nb - 1) {
            const uint32_t p = end > 0xffffffffull ? 0xffffffffu : (uint32_t)end;
            *total = p;
            host[1] = p;
        }
    }
}

// Longest tiles first: class b holds the tiles whose list length has its highest set bit at b
// (empty tiles last); within a class the order is that of the atomics (it only schedules).  One
// block of at least 33 threads.
__device__ void order_tiles(const int2* __restrict__ ranges, int tiles, int32_t* __restrict__ order) {
    __shared__ int s_cnt[33], s_pos[33];
    const int t = threadIdx.x;
    if (t < 33) s_cnt[t] = 0;
    __syncthreads();
    auto cls = [&](int i) {
        const int2 r = ranges[i];
        const int len = r.y - r.x;
        return len > 0 ? 32 - __clz(len) : 0;  // 1..31, 0 for an empty tile
    };
    for (int i = t; i < tiles; i += blockDim.x) atomicAdd(&s_cnt[cls(i)], 1);
    __syncthreads();
    if (t == 0) {
        int run = 0;
        for (int c = 32; c >= 0; --c) {
            s_pos[c] = run;
            run += s_cnt[c];
        }
    }
    __syncthreads();
    for (int i = t; i < tiles; i += blockDim.x) order[atomicAdd(&s_pos[cls(i)], 1)] = i;
}

__global__ void __launch_bounds__(1024) tile_order_kernel(const int2* __restrict__ ranges, int tiles,
                                                          int32_t* __restrict__ order) {
    order_tiles(ranges, tiles, order);
}

// Pairs into their tiles' ranges; with `order`, block 0 writes the tiles' launch order instead.
// Nothing is written past `limit` pairs or after a look-back that gave up.
__global__ void __launch_bounds__(kBinThreads) place_pairs(int N, int parts, const int32_t* __restrict__ touched,
                                                           const int4* __restrict__ rect, int tiles_x, int tiles,
                                                           const int2* __restrict__ ranges,
                                                           uint32_t* __restrict__ placed,
                                                           const uint32_t* __restrict__ total, uint32_t limit,
                                                           const uint32_t* __restrict__ err, int32_t* __restrict__ ids,
                                                           int32_t* __restrict__ order) {
    int block = blockIdx.x;
    if (order) {
        if (block == 0) {
            order_tiles(ranges, tiles, order);
            return;
        }
        --block;
    }
    if (*total > limit || *err) return;
    warp_pairs(block * (kBinThreads / 32) + (int)threadIdx.x / 32, parts, N, touched, rect, tiles_x, tiles,
               [&](int own, int t) {
                   const int2 r = ranges[t];
                   const int at = r.x + (int)atomicAdd(placed + (size_t)t * kTileWords, 1u);
                   if (at < r.y) ids[at] = own;
               });
}

// Per-tile depth order.  Each list is sorted on the 64-bit key (binary32 depth bits, index), i.e.
// by depth with ties in index order (visible depths are > z_near > 0, so their bits order like
// the values).  In a list of up to kTsThreads keys (distinct, by their index) every thread counts
// the keys below its own, which is its place: one pass of broadcast reads with no barrier instead
// of up to 36 network steps (83,000 pairs in 1,200 tiles 18.1 -> 16.8 us, 251,000 in 3,225 32.4 ->
// 22.8, 890 in 12 10.5 -> 6.5, launch included; counting up to 128 keys only: 16.8, 24.1, 10.2).
// Lists of up to kTsCap keys are sorted in shared memory by a bitonic network; longer ones are cut into
// kTsCap runs sorted the same way and merged pairwise through the scratch buffers (two arrays of
// `scratch` keys, each tile using its own segment; with more pairs than that they are left for a
// second launch with larger ones).  Lists of up to `longer` keys are left as they are.  A binning that
// failed (*err) or does not fit leaves every tile empty.
constexpr int kTsThreads = 256;
constexpr int kTsCap = 4096;

__device__ __forceinline__ uint64_t depth_index_key(const float* __restrict__ depth, uint32_t g) {
    return ((uint64_t)__float_as_uint(depth[g]) << 32) | g;
}

// Bitonic sort of s[0, n2) (n2 a power of two) by the whole block, ascending.  Pair p of a step
// with stride j works on i = p with a zero bit inserted at j and i + j, so that the 32 pairs of a
// warp stay within their own 64 keys while j <= 32 and need no block barrier between such steps.
__device__ void block_bitonic(uint64_t* s, int n2) {
    for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int p = threadIdx.x; p < n2 / 2; p += blockDim.x) {
                const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1));
                const uint64_t a = s[i], b = s[i + j];
                if ((a > b) == ((i & k) == 0)) {
                    s[i] = b;
                    s[i + j] = a;
                }
            }
            // the next step's stride: j / 2, or k at the start of the next merge
            if (j > 32 || (j > 1 ? j / 2 : k) > 32)
                __syncthreads();
            else
                __syncwarp();
        }
    __syncthreads();
}

// Number of elements taken from a (length na) among the first `diag` outputs of the merge of
// a and b (length nb): the merge-path split, ties taken from a first.
__device__ __forceinline__ int merge_split(const uint64_t* a, int na, const uint64_t* b, int nb, int diag) {
    int lo = max(0, diag - nb), hi = min(diag, na);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] <= b[diag - 1 - mid]) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(kTsThreads) tile_depth_sort(int2* __restrict__ ranges,
                                                              const float* __restrict__ depth,
                                                              int32_t* __restrict__ ids, uint64_t* __restrict__ buf0,
                                                              uint64_t* __restrict__ buf1, uint32_t scratch, int longer,
                                                              const uint32_t* __restrict__ total, uint32_t limit,
                                                              const uint32_t* __restrict__ err) {
    __shared__ __align__(16) uint64_t s[kTsCap];
    const uint32_t P = *total;
    if (*err || P > limit) {
        if (threadIdx.x == 0) ranges[blockIdx.x] = make_int2(0, 0);
        return;
    }
    const int2 r = ranges[blockIdx.x];
    const int L = r.y - r.x;
    if (L == 0 && threadIdx.x == 0) ranges[blockIdx.x] = make_int2(0, 0);
    if (L <= longer) return;
    int32_t* list = ids + r.x;
    if (L <= kTsThreads) {
        const int t = threadIdx.x;
        if (t < ((L + 1) & ~1)) s[t] = t < L ? depth_index_key(depth, (uint32_t)list[t]) : ~0ull;
        __syncthreads();
        if (t < L) {
            const uint64_t own = s[t];
            int rank = 0;
#pragma unroll 4
            for (int j = 0; j < L; j += 2) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + j);
                rank += (v.x < own) + (v.y < own);
            }
            list[rank] = (int32_t)(uint32_t)own;
        }
        return;
    }
    if (L <= kTsCap) {
        int n2 = 1;
        while (n2 < L) n2 <<= 1;
        for (int i = threadIdx.x; i < n2; i += blockDim.x)
            s[i] = i < L ? depth_index_key(depth, (uint32_t)list[i]) : ~0ull;
        __syncthreads();
        block_bitonic(s, n2);
        for (int i = threadIdx.x; i < L; i += blockDim.x) list[i] = (int32_t)(uint32_t)s[i];
        return;
    }
    if (P > scratch) return;
    // long list: sorted runs of kTsCap keys, then pairwise merges
    uint64_t* src = buf0 + r.x;
    uint64_t* dst = buf1 + r.x;
    for (int c0 = 0; c0 < L; c0 += kTsCap) {
        const int n = min(kTsCap, L - c0);
        for (int i = threadIdx.x; i < kTsCap; i += blockDim.x)
            s[i] = i < n ? depth_index_key(depth, (uint32_t)list[c0 + i]) : ~0ull;
        __syncthreads();
        block_bitonic(s, kTsCap);
        for (int i = threadIdx.x; i < n; i += blockDim.x) src[c0 + i] = s[i];
        __syncthreads();
    }
    for (int width = kTsCap; width < L; width <<= 1) {
        for (int m0 = 0; m0 < L; m0 += 2 * width) {
            const int na = min(width, L - m0), nb = max(0, min(width, L - m0 - width));
            const uint64_t* a = src + m0;
            const uint64_t* b = a + na;
            const int total_ab = na + nb;
            const int per = (total_ab + blockDim.x - 1) / blockDim.x;
            const int d0 = min(total_ab, (int)threadIdx.x * per), d1 = min(total_ab, d0 + per);
            int ia = merge_split(a, na, b, nb, d0), ib = d0 - ia;
            for (int o = d0; o < d1; ++o) {
                const bool take_a = ib >= nb || (ia < na && a[ia] <= b[ib]);
                dst[m0 + o] = take_a ? a[ia++] : b[ib++];
            }
        }
        __syncthreads();
        uint64_t* t = src;
        src = dst;
        dst = t;
    }
    for (int i = threadIdx.x; i < L; i += blockDim.x) list[i] = (int32_t)(uint32_t)src[i];
}

// Counters of binning slot k (a keyframe of a batch; a single binning uses slot 0): on the
// device 4 words at cnt + 16 k ([1] the pair count P, [2] the error word of a look-back that gave
// up), written to 4 pinned host words at host_counts + 8 + 4 k with the tensor-core wait flag, and
// the event that says they have been written.
struct BinSlot {
    uint32_t *cnt, *host;
    cudaEvent_t counted;
    void* words;
    uint64_t* lng;
    uint32_t lng_keys;  // keys of each of the two merge buffers
};

constexpr size_t kLongKeys = 1 << 18;  // merge scratch held from the start: keys per buffer

// Scratch buffer j of binning slot k (j: 0 counters, 1 long-list merge buffers): slot 0 uses the
// context's workspace slots, the others their own buffers, so that the keyframes of a batch can be
// binned at the same time.
void* bin_scratch(latentam_ctx* ctx, int slot, int j, size_t bytes) {
    if (slot == 0) return ws(ctx, j == 0 ? WS_BIN_WORDS : WS_BIN_LONG, bytes);
    return frame_ws(ctx, 2 * LATENTAM_MAX_BATCH + 2 * slot + j, bytes);
}
size_t bin_scratch_bytes(const latentam_ctx* ctx, int slot, int j) {
    return slot == 0 ? ctx->slot_bytes[j == 0 ? WS_BIN_WORDS : WS_BIN_LONG]
                     : ctx->frame_bytes[2 * LATENTAM_MAX_BATCH + 2 * slot + j];
}

latentam_status bin_slot(latentam_ctx* ctx, int slot, int64_t tiles, BinSlot* b) {
    if (slot < 0 || slot >= LATENTAM_MAX_BATCH) {
        set_error("binning slot %d outside 0..%d", slot, LATENTAM_MAX_BATCH - 1);
        return LATENTAM_ERR_INVALID_ARG;
    }
    uint32_t* c = static_cast<uint32_t*>(ws(ctx, WS_COUNTERS, 64 * LATENTAM_MAX_BATCH));
    b->words = bin_scratch(ctx, slot, 0, bin_words_bytes(tiles));
    b->lng = static_cast<uint64_t*>(bin_scratch(ctx, slot, 1, 16 * kLongKeys));
    if (!c || !b->words || !b->lng) return LATENTAM_ERR_OUT_OF_MEMORY;
    b->lng_keys = (uint32_t)std::min<size_t>(bin_scratch_bytes(ctx, slot, 1) / 16, (size_t)kMaxPairs);
    b->cnt = c + 16 * slot;
    b->host = ctx->host_counts + 8 + 4 * slot;
    cudaEvent_t& ev = ctx->count_events[slot];
    if (!ev) {
        cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return cuda_error(e, "binning event");
    }
    b->counted = ev;
    return LATENTAM_OK;
}

uint32_t pair_limit(const latentam_bins& bins) {
    return (uint32_t)std::min<int64_t>(bins.capacity, kMaxPairs);
}

}  // namespace

latentam_status launch_tile_order(const CamParams& cam, const latentam_bins& bins, int32_t* order, cudaStream_t st) {
    const int tiles = cam.tiles_x * cam.tiles_y;
    tile_order_kernel<<<1, 1024, 0, st>>>(reinterpret_cast<const int2*>(bins.tile_ranges), tiles, order);
    LAT_CHECK_LAUNCH("tile_order_kernel");
    return LATENTAM_OK;
}

latentam_status bin_launch(latentam_ctx* ctx, int32_t N, const latentam_projected& proj, const CamParams& cam,
                           const latentam_bins& bins, int32_t* order, int slot, cudaStream_t st) {
    const int64_t num_tiles = (int64_t)cam.tiles_x * cam.tiles_y;
    const int tiles = (int)num_tiles;
    int2* ranges = reinterpret_cast<int2*>(bins.tile_ranges);
    if (N == 0) {
        cudaError_t e = cudaMemsetAsync(ranges, 0, sizeof(int2) * (size_t)num_tiles, st);
        if (e != cudaSuccess) return cuda_error(e, "memset tile_ranges");
        return order ? launch_tile_order(cam, bins, order, st) : LATENTAM_OK;
    }
    BinSlot b;
    LAT_TRY(bin_slot(ctx, slot, num_tiles, &b));
    const BinWords w = bin_words(b.words, num_tiles);
    const int nb = (tiles + kScanTiles - 1) / kScanTiles;
    const int parts = pair_parts(N, ctx->num_sms);
    const unsigned blocks = (unsigned)((((int64_t)N + 31) / 32 * parts + kBinThreads / 32 - 1) / (kBinThreads / 32));
    const int4* rect = reinterpret_cast<const int4*>(proj.rect);
    // an armed test stall applies to the last block of the scan (once)
    const bool stall = ctx->test_stall_sort && nb > 1;
    // Both halves replay a captured graph once the same frame size and buffers recur; nothing in
    // them depends on the pair count.
    auto count = [&](cudaStream_t s) -> latentam_status {
        cudaError_t e = cudaMemsetAsync(b.words, 0, bin_words_bytes(num_tiles), s);
        if (e != cudaSuccess) return cuda_error(e, "clear the binning counters");
        count_tiles<<<blocks, kBinThreads, 0, s>>>(N, parts, proj.tiles_touched, rect, cam.tiles_x, tiles, w.count, b.cnt + 2,
                                                   ctx->dev_flags, b.host);
        LAT_CHECK_LAUNCH("count_tiles");
        tile_scan<<<nb, kScanTiles, 0, s>>>(w, tiles, ranges, b.cnt + 1, b.host, b.cnt + 2,
                                            stall ? kTestSpinLimit : kSpinLimit, stall ? nb - 1 : -1);
        LAT_CHECK_LAUNCH("tile_scan");
        return LATENTAM_OK;
    };
    const uint64_t ckey[] = {0x62696e302d636e74ull /* tag: counting */, (uint64_t)N, (uint64_t)num_tiles,
                             (uint64_t)cam.tiles_x, reinterpret_cast<uint64_t>(proj.tiles_touched),
                             reinterpret_cast<uint64_t>(proj.rect), reinterpret_cast<uint64_t>(ranges),
                             reinterpret_cast<uint64_t>(b.host), reinterpret_cast<uint64_t>(b.words),
                             reinterpret_cast<uint64_t>(st), ctx->ws_generation, (uint64_t)stall};
    LAT_TRY(cached_launch(ctx, ckey, (int)(sizeof(ckey) / sizeof(ckey[0])), st, count));
    if (stall) ctx->test_stall_sort = 0;
    cudaError_t e = cudaEventRecord(b.counted, st);
    if (e != cudaSuccess) return cuda_error(e, "record the pair count");
    const uint32_t limit = pair_limit(bins);
    auto place = [&](cudaStream_t s) -> latentam_status {
        place_pairs<<<blocks + (order ? 1 : 0), kBinThreads, 0, s>>>(N, parts, proj.tiles_touched, rect, cam.tiles_x, tiles,
                                                                     ranges, w.placed, b.cnt + 1, limit, b.cnt + 2,
                                                                     bins.pair_ids, order);
        LAT_CHECK_LAUNCH("place_pairs");
        tile_depth_sort<<<(unsigned)tiles, kTsThreads, 0, s>>>(ranges, proj.depth, bins.pair_ids, b.lng,
                                                               b.lng + b.lng_keys, b.lng_keys, 1, b.cnt + 1, limit,
                                                               b.cnt + 2);
        LAT_CHECK_LAUNCH("tile_depth_sort");
        return LATENTAM_OK;
    };
    const uint64_t pkey[] = {0x62696e312d706c63ull /* tag: placing */, (uint64_t)N, (uint64_t)num_tiles,
                             (uint64_t)cam.tiles_x, (uint64_t)limit, reinterpret_cast<uint64_t>(proj.depth),
                             reinterpret_cast<uint64_t>(proj.tiles_touched), reinterpret_cast<uint64_t>(proj.rect),
                             reinterpret_cast<uint64_t>(bins.pair_ids), reinterpret_cast<uint64_t>(ranges),
                             reinterpret_cast<uint64_t>(b.cnt), reinterpret_cast<uint64_t>(b.words),
                             reinterpret_cast<uint64_t>(b.lng), reinterpret_cast<uint64_t>(order),
                             reinterpret_cast<uint64_t>(st), ctx->ws_generation};
    return cached_launch(ctx, pkey, (int)(sizeof(pkey) / sizeof(pkey[0])), st, place);
}

latentam_status bin_wait(latentam_ctx* ctx, int32_t N, const latentam_projected& proj, const CamParams& cam,
                         latentam_bins* bins, int slot, cudaStream_t st) {
    if (N == 0) {
        bins->num_pairs = 0;
        return LATENTAM_OK;
    }
    const int64_t num_tiles = (int64_t)cam.tiles_x * cam.tiles_y;
    BinSlot b;
    LAT_TRY(bin_slot(ctx, slot, num_tiles, &b));
    cudaError_t e = cudaEventSynchronize(b.counted);
    if (e != cudaSuccess) return cuda_error(e, "wait for the pair count");
    volatile uint32_t* host = b.host;
    const uint32_t sort_error = host[2], tc_error = host[3];
    const int64_t P = (int64_t)host[1];
    if (sort_error) {
        e = cudaMemsetAsync(b.cnt + 2, 0, sizeof(uint32_t), st);
        if (e != cudaSuccess) return cuda_error(e, "clear the binning error word");
        set_error("a binning look-back wait gave up in an earlier binning (its tiles were left empty)");
        return LATENTAM_ERR_TIMEOUT;
    }
    if (tc_error) {
        host[3] = 0;  // reported once, by this slot
        e = cudaMemsetAsync(ctx->dev_flags, 0, sizeof(int), st);
        if (e != cudaSuccess) return cuda_error(e, "clear the tensor-core wait flag");
        set_error("a bounded wait of a tensor-core decode kernel gave up in an earlier call (its loss was NaN)");
        return LATENTAM_ERR_TIMEOUT;
    }
    bins->num_pairs = P;
    if (P > bins->capacity) {
        set_error("pair buffer holds %lld pairs, %lld needed", (long long)bins->capacity, (long long)P);
        return LATENTAM_ERR_CAPACITY;
    }
    if (P > kMaxPairs) {
        set_error("binning of %lld pairs is not supported", (long long)P);
        return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
    if (P > (int64_t)b.lng_keys) {
        // lists too long for shared memory found no room in the merge buffers: sort those with larger ones
        uint64_t* lng = static_cast<uint64_t*>(bin_scratch(ctx, slot, 1, 16 * (size_t)P));
        if (!lng) return LATENTAM_ERR_OUT_OF_MEMORY;
        tile_depth_sort<<<(unsigned)num_tiles, kTsThreads, 0, st>>>(reinterpret_cast<int2*>(bins->tile_ranges),
                                                                    proj.depth, bins->pair_ids, lng, lng + P,
                                                                    (uint32_t)P, kTsCap, b.cnt + 1, pair_limit(*bins),
                                                                    b.cnt + 2);
        LAT_CHECK_LAUNCH("tile_depth_sort");
    }
    return LATENTAM_OK;
}

latentam_status bin_and_sort(latentam_ctx* ctx, int32_t N, const latentam_projected& proj, const CamParams& cam,
                             latentam_bins* bins, int32_t* order, cudaStream_t st) {
    LAT_TRY(bin_launch(ctx, N, proj, cam, *bins, order, 0, st));
    return bin_wait(ctx, N, proj, cam, bins, 0, st);
}

}  // namespace lat

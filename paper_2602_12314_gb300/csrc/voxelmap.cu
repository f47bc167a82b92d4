// Voxel-hashed global map and the active local map around the camera (Sec. III-E, "Local-
// Global Map Management via Voxel Hashing").
//
// The global store (Gaussian attributes in index order) and its slot table live in HBM: at
// 172 bytes per Gaussian (d = 32) the 280 GB of a GB300 hold on the order of 10^9 of them, so
// the radius gather, the de-duplication and the write-back run as kernels instead of host loops.
// Each Gaussian owns the slot of the voxel floor(p / s_v) it was inserted from; slots hold no key
// (two voxels with the same hash collide and the later one counts as occupied), at most one
// Gaussian per slot.  Insert-if-free is deterministic: every candidate whose slot is empty claims
// it with an atomic minimum of its input index, the lowest index wins, and the winners are
// appended in input order (an exclusive scan), exactly as a sequential insertion would.
//
// Synchronisation: Local -> Global (local Gaussians that came from the store overwrite their
// entries, new ones are inserted if their slot is free), then Global -> Local (local Gaussians
// outside the radius are dropped, kept ones are marked in a per-row epoch array, and the store's
// unmarked Gaussians inside the radius are appended in index order) into the second of two local
// buffers.  The local map also carries the Adam moments of the queries (zero for appended rows).
#include <algorithm>
#include <climits>
#include <cstring>

#include "internal.cuh"

using namespace lat;

namespace {

constexpr int kMapThreads = 256;
constexpr int64_t kMaxInsert = 1ll << 24;  // rows of one insertion

struct Rows {  // SoA rows of Gaussians (any may be null where not used)
    float *means, *quats, *scales, *opac, *f, *m_f, *v_f;
    int32_t* gidx;
    bool host;  // pinned host memory (read and written by the kernels through unified addressing)
};

}  // namespace

struct latentam_map {
    int device;
    int d;
    int table_log2;
    float voxel_size;
    int64_t capacity, count;  // global store (count mirrored on the host)
    bool host_store;          // the store's rows in pinned host memory
    int32_t* table;           // 2^table_log2 slots, -1 = empty
    int32_t* claim;           // per-slot claims of one insertion, INT_MAX when idle
    int32_t* epoch_mark;      // per global row: the last synchronisation that found it local
    int32_t epoch;
    Rows g;
    Rows loc[2];
    int64_t loc_capacity[2];
    int cur;                  // the current local buffer
    int64_t local_count;
    bool fresh;               // rows were added, or the last synchronisation met rows without a store
                              // entry: the next one inserts first
    // scratch of one operation: slots and candidate flags per row, kept / selected rows per block
    int32_t* slot;
    uint32_t *flag, *pos;
    int64_t scratch_n;
    uint32_t* total;          // device counters (3) and their pinned copy
    uint32_t* host_total;
};

namespace {

void free_rows(Rows& r) {
    for (void* p : {(void*)r.means, (void*)r.quats, (void*)r.scales, (void*)r.opac, (void*)r.f, (void*)r.m_f,
                    (void*)r.v_f, (void*)r.gidx})
        if (p) {
            if (r.host) cudaFreeHost(p);
            else cudaFree(p);
        }
    r = Rows{};
}

// Rows of `cap` Gaussians (moments and gidx only when `local`); the first `keep` rows of `old`
// are copied over and `old` is freed.
latentam_status alloc_rows(Rows& r, int64_t cap, int d, bool local, Rows* old, int64_t keep, bool host = false) {
    Rows n{};
    n.host = host;
    auto alloc = [&](void** p, size_t bytes) {
        return host ? cudaHostAlloc(p, bytes, cudaHostAllocMapped) : cudaMalloc(p, bytes);
    };
    const size_t c = (size_t)std::max<int64_t>(cap, 1);
    struct Field {
        float** dst;
        float* src;
        int w;
    } fields[] = {{&n.means, old ? old->means : nullptr, 3},  {&n.quats, old ? old->quats : nullptr, 4},
                  {&n.scales, old ? old->scales : nullptr, 3}, {&n.opac, old ? old->opac : nullptr, 1},
                  {&n.f, old ? old->f : nullptr, d},           {&n.m_f, old ? old->m_f : nullptr, local ? d : 0},
                  {&n.v_f, old ? old->v_f : nullptr, local ? d : 0}};
    for (auto& fl : fields) {
        if (fl.w == 0) continue;
        if (alloc(reinterpret_cast<void**>(fl.dst), sizeof(float) * c * fl.w) != cudaSuccess) {
            cudaGetLastError();
            free_rows(n);
            set_error("voxel map: out of device memory for %lld rows", (long long)cap);
            return LATENTAM_ERR_OUT_OF_MEMORY;
        }
        if (fl.src && keep > 0) cudaMemcpy(*fl.dst, fl.src, sizeof(float) * (size_t)keep * fl.w, cudaMemcpyDefault);
    }
    if (local) {
        if (cudaMalloc(&n.gidx, sizeof(int32_t) * c) != cudaSuccess) {
            cudaGetLastError();
            free_rows(n);
            set_error("voxel map: out of device memory for %lld rows", (long long)cap);
            return LATENTAM_ERR_OUT_OF_MEMORY;
        }
        if (old && old->gidx && keep > 0)
            cudaMemcpy(n.gidx, old->gidx, sizeof(int32_t) * (size_t)keep, cudaMemcpyDeviceToDevice);
    }
    if (old) free_rows(*old);
    r = n;
    return LATENTAM_OK;
}

latentam_status grow_global(latentam_map* m, int64_t need) {
    if (need <= m->capacity) return LATENTAM_OK;
    if (need > INT32_MAX) {
        set_error("voxel map: %lld Gaussians exceed the int32 indices", (long long)need);
        return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
    const int64_t cap = std::min<int64_t>(INT32_MAX, std::max<int64_t>(need, 2 * m->capacity));
    cudaDeviceSynchronize();
    Rows old = m->g;
    LAT_TRY(alloc_rows(m->g, cap, m->d, false, &old, m->count, m->host_store));
    int32_t* mark = nullptr;
    if (cudaMalloc(&mark, sizeof(int32_t) * (size_t)cap) != cudaSuccess) {
        cudaGetLastError();
        set_error("voxel map: out of device memory");
        return LATENTAM_ERR_OUT_OF_MEMORY;
    }
    cudaMemset(mark, 0, sizeof(int32_t) * (size_t)cap);
    if (m->epoch_mark) {
        cudaMemcpy(mark, m->epoch_mark, sizeof(int32_t) * (size_t)m->count, cudaMemcpyDeviceToDevice);
        cudaFree(m->epoch_mark);
    }
    m->epoch_mark = mark;
    m->capacity = cap;
    return LATENTAM_OK;
}

latentam_status grow_local(latentam_map* m, int which, int64_t need, int64_t keep) {
    if (need <= m->loc_capacity[which]) return LATENTAM_OK;
    const int64_t cap = std::max<int64_t>(need, 2 * m->loc_capacity[which]);
    cudaDeviceSynchronize();
    Rows old = m->loc[which];
    LAT_TRY(alloc_rows(m->loc[which], cap, m->d, true, &old, keep));
    m->loc_capacity[which] = cap;
    return LATENTAM_OK;
}

latentam_status grow_scratch(latentam_map* m, int64_t n) {
    if (n <= m->scratch_n) return LATENTAM_OK;
    const int64_t cap = std::max<int64_t>(n, 2 * m->scratch_n);
    cudaDeviceSynchronize();
    if (m->slot) cudaFree(m->slot);
    if (m->flag) cudaFree(m->flag);
    if (m->pos) cudaFree(m->pos);
    m->slot = nullptr, m->flag = m->pos = nullptr;
    if (cudaMalloc(&m->slot, sizeof(int32_t) * (size_t)cap) != cudaSuccess ||
        cudaMalloc(&m->flag, sizeof(uint32_t) * (size_t)cap) != cudaSuccess ||
        cudaMalloc(&m->pos, sizeof(uint32_t) * (size_t)cap) != cudaSuccess) {
        cudaGetLastError();
        set_error("voxel map: out of device memory for scratch");
        return LATENTAM_ERR_OUT_OF_MEMORY;
    }
    m->scratch_n = cap;
    return LATENTAM_OK;
}

// ---- device arithmetic (every rounding explicit: the oracle takes the same decisions) -------

__device__ __forceinline__ int slot_of(float x, float y, float z, float s_v, int table_log2) {
    const int64_t vx = (int64_t)floorf(__fdiv_rn(x, s_v)), vy = (int64_t)floorf(__fdiv_rn(y, s_v)),
                  vz = (int64_t)floorf(__fdiv_rn(z, s_v));
    const uint64_t h = ((uint64_t)vx * 73856093ull) ^ ((uint64_t)vy * 19349663ull) ^ ((uint64_t)vz * 83492791ull);
    return (int)(h & ((1ull << table_log2) - 1ull));
}

__device__ __forceinline__ bool in_radius(const float* p, float cx, float cy, float cz, float r2) {
    const float dx = __fsub_rn(p[0], cx), dy = __fsub_rn(p[1], cy), dz = __fsub_rn(p[2], cz);
    const float s = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
    return s <= r2;
}

// ---- row movement ---------------------------------------------------------------------------
//
// A block looks at kMapThreads consecutive rows, lists the ones it moves in shared memory and copies
// them element by element, so that neighbouring threads touch neighbouring words (a thread per
// row left every 172- or 432-byte row to one thread's scattered words: 109 us to compact 111,000
// local rows of d = 32, 96 MB, against 22 us).  Bound by HBM: each row read and written once.

struct RowList {
    int32_t src[kMapThreads];   // row, counted from the block's first
    int64_t dst[kMapThreads];
    int32_t warp[kMapThreads / 32];
};

// Lists the rows with `take` in order (every thread of the block); returns their number.  With
// first >= 0 they go to consecutive rows from there, else each to its thread's `to`.
__device__ __forceinline__ int list_rows(RowList& l, bool take, int64_t first, int64_t to) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t vote = __ballot_sync(0xffffffffu, take);
    if (lane == 0) l.warp[warp] = __popc(vote);
    __syncthreads();
    int at = __popc(vote & ((1u << lane) - 1u)), n = 0;
#pragma unroll
    for (int w = 0; w < kMapThreads / 32; ++w) {
        if (w < warp) at += l.warp[w];
        n += l.warp[w];
    }
    if (take) {
        l.src[at] = threadIdx.x;
        l.dst[at] = first >= 0 ? first + at : to;
    }
    __syncthreads();
    return n;
}

template <class T>
__device__ __forceinline__ void move_field(const RowList& l, int n, int64_t i0, uint32_t w, const T* __restrict__ s,
                                           T* __restrict__ t) {
#pragma unroll 4
    for (uint32_t e = threadIdx.x; e < (uint32_t)n * w; e += kMapThreads) {
        const uint32_t r = e / w, k = e - r * w;
        t[l.dst[r] * w + k] = s[(i0 + l.src[r]) * w + k];
    }
}

enum class Moments { kNone, kCopy, kZero };

// The listed rows of s (counted from i0) to t.  vec: d is a multiple of 4 and the d-wide arrays
// are 16-byte aligned.
template <Moments MO>
__device__ __forceinline__ void move_rows(const RowList& l, int n, int64_t i0, const Rows& s, const Rows& t, int d,
                                          bool vec) {
    move_field(l, n, i0, 3, s.means, t.means);
    move_field(l, n, i0, 4, s.quats, t.quats);
    move_field(l, n, i0, 3, s.scales, t.scales);
    move_field(l, n, i0, 1, s.opac, t.opac);
    if (vec) {
        const uint32_t w = (uint32_t)d / 4;
        auto v4 = [](float* p) { return reinterpret_cast<float4*>(p); };
        move_field<float4>(l, n, i0, w, v4(s.f), v4(t.f));
        if (MO == Moments::kCopy) {
            move_field<float4>(l, n, i0, w, v4(s.m_f), v4(t.m_f));
            move_field<float4>(l, n, i0, w, v4(s.v_f), v4(t.v_f));
        }
    } else {
        move_field(l, n, i0, (uint32_t)d, s.f, t.f);
        if (MO == Moments::kCopy) {
            move_field(l, n, i0, (uint32_t)d, s.m_f, t.m_f);
            move_field(l, n, i0, (uint32_t)d, s.v_f, t.v_f);
        }
    }
    if (MO == Moments::kZero)
        for (uint32_t e = threadIdx.x; e < (uint32_t)n * d; e += kMapThreads) {
            const uint32_t r = e / d, k = e - r * d;
            t.m_f[l.dst[r] * d + k] = t.v_f[l.dst[r] * d + k] = 0.f;
        }
}

bool vec_rows(int d, const Rows& s, const Rows& t) {
    uintptr_t a = 0;
    for (const float* p : {s.f, s.m_f, s.v_f, t.f, t.m_f, t.v_f}) a |= reinterpret_cast<uintptr_t>(p);
    return d % 4 == 0 && (a & 15u) == 0;
}

// In-place exclusive scans of up to two lists of block counts (block b takes list b) and their
// totals; 4096 counts at a time with a carry.
__global__ void __launch_bounds__(1024) scan_counts(uint32_t* a, int64_t na, uint32_t* b, int64_t nb,
                                                    uint32_t* __restrict__ total) {
    __shared__ uint32_t s_warp[32], s_carry;
    uint32_t* v = blockIdx.x ? b : a;
    const int64_t n = blockIdx.x ? nb : na;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += 4096) {
        uint32_t x[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = base + 4 * t + k;
            x[k] = i < n ? v[i] : 0u;
            sum += x[k];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        uint32_t run = s_carry + incl - sum, all = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < warp) run += s_warp[w];
            all += s_warp[w];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = base + 4 * t + k;
            if (i < n) v[i] = run;
            run += x[k];
        }
        __syncthreads();
        if (t == 0) s_carry += all;
        __syncthreads();
    }
    if (t == 0) total[blockIdx.x] = s_carry;
}

// Candidates: rows whose slot is empty (and, with gidx, that have no global entry yet) claim it.
__global__ void insert_claim(int64_t n, const float* __restrict__ means, const int32_t* __restrict__ gidx,
                             float s_v, int table_log2, const int32_t* __restrict__ table, int32_t* claim,
                             int32_t* __restrict__ slot, uint32_t* __restrict__ cand) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int s = -1;
    uint32_t c = 0;
    if (!gidx || gidx[i] < 0) {
        s = slot_of(means[3 * i], means[3 * i + 1], means[3 * i + 2], s_v, table_log2);
        if (table[s] < 0) {
            c = 1;
            atomicMin(claim + s, (int)i);
        }
    }
    slot[i] = s;
    cand[i] = c;
}

// cand[i] = 1 where candidate i holds the lowest claim of its slot, 2 where it lost; won[block] =
// the block's winners.
__global__ void __launch_bounds__(kMapThreads) insert_win(int64_t n, const int32_t* __restrict__ slot,
                                                          const int32_t* __restrict__ claim, uint32_t* cand,
                                                          uint32_t* __restrict__ won) {
    const int64_t i = (int64_t)blockIdx.x * kMapThreads + threadIdx.x;
    bool w = false;
    if (i < n && cand[i]) {
        w = claim[slot[i]] == (int32_t)i;
        cand[i] = w ? 1u : 2u;
    }
    const int c = __syncthreads_count(w);
    if (threadIdx.x == 0) won[blockIdx.x] = (uint32_t)c;
}

// Winners take the indices from base on, in input order (won: the scanned block counts), and their
// slot; every claim is released.
__global__ void __launch_bounds__(kMapThreads) insert_commit(int64_t n, Rows src, int d, bool vec,
                                                             const int32_t* __restrict__ slot,
                                                             const uint32_t* __restrict__ cand,
                                                             const uint32_t* __restrict__ won, int64_t base,
                                                             int32_t* table, int32_t* claim, Rows dst,
                                                             int32_t* __restrict__ out_index,
                                                             int32_t* __restrict__ gidx_out) {
    __shared__ RowList l;
    const int64_t i0 = (int64_t)blockIdx.x * kMapThreads, i = i0 + threadIdx.x;
    const uint32_t w = i < n ? cand[i] : 0u;
    if (w) claim[slot[i]] = INT_MAX;
    const int cnt = list_rows(l, w == 1, base + won[blockIdx.x], 0);
    if (out_index && i < n && w != 1) out_index[i] = -1;
    if ((int)threadIdx.x < cnt) {
        const int64_t r = i0 + l.src[threadIdx.x];
        const int32_t idx = (int32_t)l.dst[threadIdx.x];
        table[slot[r]] = idx;
        if (gidx_out) gidx_out[r] = idx;
        if (out_index) out_index[r] = idx;
    }
    move_rows<Moments::kNone>(l, cnt, i0, src, dst, d, vec);
}

// Local -> Global for the rows with a store entry, and the first half of the prune: kept[block] =
// the block's local rows inside the radius, whose store entries are marked with the epoch.  A row
// without an entry leaves the epoch in *unstored.
__global__ void __launch_bounds__(kMapThreads) write_back(int64_t n, Rows local, int d, bool vec, Rows global,
                                                          float cx, float cy, float cz, float r2,
                                                          int32_t* __restrict__ epoch_mark, int32_t epoch,
                                                          uint32_t* __restrict__ kept, uint32_t* unstored) {
    __shared__ RowList l;
    const int64_t i0 = (int64_t)blockIdx.x * kMapThreads, i = i0 + threadIdx.x;
    const int32_t g = i < n ? local.gidx[i] : -1;
    const bool k = i < n && in_radius(local.means + 3 * i, cx, cy, cz, r2);
    if (k && g >= 0) epoch_mark[g] = epoch;
    if (i < n && g < 0) *unstored = (uint32_t)epoch;
    const int c = __syncthreads_count(k);
    if (threadIdx.x == 0) kept[blockIdx.x] = (uint32_t)c;
    const int cnt = list_rows(l, g >= 0, -1, g);
    move_rows<Moments::kNone>(l, cnt, i0, local, global, d, vec);
}

// The kept local rows to consecutive rows of the other local buffer (kept: scanned block counts).
__global__ void __launch_bounds__(kMapThreads) compact_local(int64_t n, Rows src, int d, bool vec, float cx, float cy,
                                                             float cz, float r2, const uint32_t* __restrict__ kept,
                                                             Rows dst) {
    __shared__ RowList l;
    const int64_t i0 = (int64_t)blockIdx.x * kMapThreads, i = i0 + threadIdx.x;
    const bool k = i < n && in_radius(src.means + 3 * i, cx, cy, cz, r2);
    const int cnt = list_rows(l, k, kept[blockIdx.x], 0);
    move_rows<Moments::kCopy>(l, cnt, i0, src, dst, d, vec);
    if ((int)threadIdx.x < cnt) dst.gidx[l.dst[threadIdx.x]] = src.gidx[i0 + l.src[threadIdx.x]];
}

__device__ __forceinline__ bool selected(int64_t g, int64_t n, const float* means, float cx, float cy, float cz,
                                         float r2, const int32_t* epoch_mark, int32_t epoch) {
    return g < n && in_radius(means + 3 * g, cx, cy, cz, r2) && epoch_mark[g] != epoch;
}

// sel[block] = the block's store rows inside the radius that are not local.
__global__ void __launch_bounds__(kMapThreads) select_global(int64_t n, const float* __restrict__ means, float cx,
                                                             float cy, float cz, float r2,
                                                             const int32_t* __restrict__ epoch_mark, int32_t epoch,
                                                             uint32_t* __restrict__ sel) {
    const int64_t g = (int64_t)blockIdx.x * kMapThreads + threadIdx.x;
    const int c = __syncthreads_count(selected(g, n, means, cx, cy, cz, r2, epoch_mark, epoch));
    if (threadIdx.x == 0) sel[blockIdx.x] = (uint32_t)c;
}

// Those rows appended to the local buffer from row `base` on, in index order (sel: scanned block
// counts, total: their sum).
__global__ void __launch_bounds__(kMapThreads) append_global(int64_t n, Rows global, int d, bool vec, float cx,
                                                             float cy, float cz, float r2,
                                                             const int32_t* __restrict__ epoch_mark, int32_t epoch,
                                                             const uint32_t* __restrict__ sel, uint32_t total,
                                                             int64_t base, Rows dst) {
    __shared__ RowList l;
    const uint32_t first = sel[blockIdx.x];
    if (first == (blockIdx.x + 1 < gridDim.x ? sel[blockIdx.x + 1] : total)) return;  // none of the block's rows
    const int64_t i0 = (int64_t)blockIdx.x * kMapThreads, g = i0 + threadIdx.x;
    const int cnt = list_rows(l, selected(g, n, global.means, cx, cy, cz, r2, epoch_mark, epoch), base + first, 0);
    move_rows<Moments::kZero>(l, cnt, i0, global, dst, d, vec);
    if ((int)threadIdx.x < cnt) dst.gidx[l.dst[threadIdx.x]] = (int32_t)(i0 + l.src[threadIdx.x]);
}

unsigned blocks(int64_t n) { return (unsigned)((n + kMapThreads - 1) / kMapThreads); }

// The first `k` device totals (after everything enqueued on st), through pinned memory.
latentam_status read_totals(latentam_map* m, int k, cudaStream_t st) {
    cudaError_t e = cudaMemcpyAsync(m->host_total, m->total, sizeof(uint32_t) * k, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? LATENTAM_OK : cuda_error(e, "voxel map: read counts");
}

// Insert-if-free of n rows of `src` (rows with gidx >= 0 skipped when gidx is given); the
// winners' new indices go to out_index (all rows, -1 for the others) and/or gidx.
latentam_status insert_rows(latentam_ctx* ctx, latentam_map* m, int64_t n, const Rows& src, int32_t* gidx,
                            int32_t* out_index, int64_t* n_inserted, cudaStream_t st) {
    if (n_inserted) *n_inserted = 0;
    if (n <= 0) return LATENTAM_OK;
    if (n > kMaxInsert) {
        set_error("voxel map: at most %lld Gaussians per insertion", (long long)kMaxInsert);
        return LATENTAM_ERR_UNSUPPORTED_SHAPE;
    }
    LAT_TRY(grow_global(m, m->count + n));
    LAT_TRY(grow_scratch(m, n));
    insert_claim<<<blocks(n), kMapThreads, 0, st>>>(n, src.means, gidx, m->voxel_size, m->table_log2, m->table,
                                                    m->claim, m->slot, m->flag);
    LAT_CHECK_LAUNCH("insert_claim");
    insert_win<<<blocks(n), kMapThreads, 0, st>>>(n, m->slot, m->claim, m->flag, m->pos);
    LAT_CHECK_LAUNCH("insert_win");
    scan_counts<<<1, 1024, 0, st>>>(m->pos, blocks(n), nullptr, 0, m->total);
    LAT_CHECK_LAUNCH("scan_counts");
    insert_commit<<<blocks(n), kMapThreads, 0, st>>>(n, src, m->d, vec_rows(m->d, src, m->g), m->slot, m->flag, m->pos,
                                                     m->count, m->table, m->claim, m->g, out_index, gidx);
    LAT_CHECK_LAUNCH("insert_commit");
    LAT_TRY(read_totals(m, 1, st));
    const uint32_t added = m->host_total[0];
    m->count += added;
    if (n_inserted) *n_inserted = added;
    return LATENTAM_OK;
}

Rows gaussian_rows(const latentam_gaussians& g, const float* f) {
    Rows r{};
    r.means = const_cast<float*>(g.means);
    r.quats = const_cast<float*>(g.quats);
    r.scales = const_cast<float*>(g.scales);
    r.opac = const_cast<float*>(g.opacities);
    r.f = const_cast<float*>(f);
    return r;
}

void fill_local(const latentam_map* m, latentam_map_local* out) {
    const Rows& r = m->loc[m->cur];
    *out = latentam_map_local{r.means, r.quats, r.scales, r.opac, r.f, r.m_f, r.v_f, r.gidx, m->local_count};
}

latentam_status enter_map(latentam_ctx* ctx, latentam_map* m) {
    if (!ctx || !m) {
        set_error("null context or map");
        return LATENTAM_ERR_INVALID_ARG;
    }
    if (m->device != ctx->device) {
        set_error("the map lives on device %d, the context on %d", m->device, ctx->device);
        return LATENTAM_ERR_INVALID_ARG;
    }
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_error(e, "cudaSetDevice");
    return LATENTAM_OK;
}

}  // namespace

extern "C" {

latentam_status latentam_map_create(latentam_ctx* ctx, int32_t d, int32_t table_log2, float voxel_size,
                                    int64_t capacity, int32_t host_store, latentam_map** out) {
    if (!ctx || !out) {
        set_error("null context or output");
        return LATENTAM_ERR_INVALID_ARG;
    }
    *out = nullptr;
    if (d < 1 || d > 256 || table_log2 < 4 || table_log2 > 30 || !(voxel_size > 0.f) || capacity < 0) {
        set_error("voxel map: d=%d table_log2=%d voxel_size=%g capacity=%lld out of range", d, table_log2,
                  (double)voxel_size, (long long)capacity);
        return LATENTAM_ERR_INVALID_ARG;
    }
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_error(e, "cudaSetDevice");
    latentam_map* m = new latentam_map();
    memset(m, 0, sizeof(*m));
    m->device = ctx->device;
    m->d = d;
    m->table_log2 = table_log2;
    m->voxel_size = voxel_size;
    m->host_store = host_store != 0;
    m->epoch = 0;
    const size_t T = (size_t)1 << table_log2;
    bool ok = cudaMalloc(&m->table, sizeof(int32_t) * T) == cudaSuccess &&
              cudaMalloc(&m->claim, sizeof(int32_t) * T) == cudaSuccess &&
              cudaMalloc(&m->total, sizeof(uint32_t) * 3) == cudaSuccess &&
              cudaMemset(m->total, 0, sizeof(uint32_t) * 3) == cudaSuccess &&
              cudaHostAlloc(&m->host_total, sizeof(uint32_t) * 3, cudaHostAllocDefault) == cudaSuccess;
    if (ok) ok = cudaMemset(m->table, 0xff, sizeof(int32_t) * T) == cudaSuccess;  // -1
    if (ok) {
        // INT_MAX in every claim: fill through a host pattern once
        int32_t* h = static_cast<int32_t*>(malloc(sizeof(int32_t) * std::min<size_t>(T, 1 << 20)));
        ok = h != nullptr;
        if (ok) {
            const size_t chunk = std::min<size_t>(T, 1 << 20);
            for (size_t i = 0; i < chunk; ++i) h[i] = INT_MAX;
            for (size_t o = 0; ok && o < T; o += chunk)
                ok = cudaMemcpy(m->claim + o, h, sizeof(int32_t) * std::min(chunk, T - o), cudaMemcpyHostToDevice) ==
                     cudaSuccess;
            free(h);
        }
    }
    latentam_status s = ok ? LATENTAM_OK : LATENTAM_ERR_OUT_OF_MEMORY;
    if (s == LATENTAM_OK) s = grow_global(m, std::max<int64_t>(capacity, 1024));
    if (s == LATENTAM_OK) s = grow_local(m, 0, 1024, 0);
    if (s == LATENTAM_OK) s = grow_local(m, 1, 1024, 0);
    if (s != LATENTAM_OK) {
        cudaGetLastError();
        latentam_map_destroy(m);
        if (s == LATENTAM_ERR_OUT_OF_MEMORY) set_error("voxel map: out of device memory");
        return s;
    }
    *out = m;
    return LATENTAM_OK;
}

latentam_status latentam_map_destroy(latentam_map* m) {
    if (!m) return LATENTAM_OK;
    cudaSetDevice(m->device);
    cudaDeviceSynchronize();
    free_rows(m->g);
    free_rows(m->loc[0]);
    free_rows(m->loc[1]);
    for (void* p : {(void*)m->table, (void*)m->claim, (void*)m->epoch_mark, (void*)m->slot, (void*)m->flag,
                    (void*)m->pos, (void*)m->total})
        if (p) cudaFree(p);
    if (m->host_total) cudaFreeHost(m->host_total);
    delete m;
    return LATENTAM_OK;
}

latentam_status latentam_map_insert(latentam_ctx* ctx, latentam_map* m, const latentam_gaussians* g, const float* f,
                                    int32_t* out_index, int64_t* n_inserted, latentam_stream stream) {
    LAT_TRY(enter_map(ctx, m));
    if (!g || g->n < 0 || (g->n > 0 && (!g->means || !g->quats || !g->scales || !g->opacities || !f))) {
        set_error("null or negative Gaussian input");
        return LATENTAM_ERR_INVALID_ARG;
    }
    return insert_rows(ctx, m, g->n, gaussian_rows(*g, f), nullptr, out_index, n_inserted, (cudaStream_t)stream);
}

latentam_status latentam_map_add_local(latentam_ctx* ctx, latentam_map* m, const latentam_gaussians* g,
                                       const float* f, latentam_stream stream) {
    LAT_TRY(enter_map(ctx, m));
    if (!g || g->n < 0 || (g->n > 0 && (!g->means || !g->quats || !g->scales || !g->opacities || !f))) {
        set_error("null or negative Gaussian input");
        return LATENTAM_ERR_INVALID_ARG;
    }
    const int64_t n = g->n;
    if (n == 0) return LATENTAM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    cudaStreamSynchronize(st);
    LAT_TRY(grow_local(m, m->cur, m->local_count + n, m->local_count));
    const Rows& L = m->loc[m->cur];
    const int64_t o = m->local_count;
    const int d = m->d;
    struct Cp {
        float* dst;
        const float* src;
        int w;
    } cps[] = {{L.means + 3 * o, g->means, 3}, {L.quats + 4 * o, g->quats, 4}, {L.scales + 3 * o, g->scales, 3},
               {L.opac + o, g->opacities, 1}, {L.f + (size_t)d * o, f, d}};
    for (auto& c : cps) {
        cudaError_t e = cudaMemcpyAsync(c.dst, c.src, sizeof(float) * (size_t)n * c.w, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return cuda_error(e, "voxel map: add local");
    }
    cudaError_t e = cudaMemsetAsync(L.m_f + (size_t)d * o, 0, sizeof(float) * (size_t)n * d, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(L.v_f + (size_t)d * o, 0, sizeof(float) * (size_t)n * d, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(L.gidx + o, 0xff, sizeof(int32_t) * (size_t)n, st);  // -1
    if (e != cudaSuccess) return cuda_error(e, "voxel map: add local");
    m->local_count += n;
    m->fresh = true;
    return LATENTAM_OK;
}

latentam_status latentam_map_sync(latentam_ctx* ctx, latentam_map* m, const float* centre, float radius,
                                  latentam_map_local* local_out, latentam_stream stream) {
    LAT_TRY(enter_map(ctx, m));
    if (!centre || !(radius >= 0.f)) {
        set_error("null centre or negative radius");
        return LATENTAM_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int d = m->d;
    const int64_t nl = m->local_count;
    const float cx = centre[0], cy = centre[1], cz = centre[2];
    const float r2 = radius * radius;
    // Local -> Global: new rows are inserted if free, known ones overwrite their entries; the prune's
    // counts and marks come with the same pass.  Global -> Local: the store's unmarked rows inside
    // the radius; one host read of both counts, then compact and append into the other buffer.
    // The insertion runs first where some rows are known to lack an entry, and is skipped elsewhere.
    // gidx is the caller's to write, so the pass looks at every row's: where it meets one without
    // an entry all the same, the rows are inserted and the pass is taken again.
    Rows local = m->loc[m->cur];
    const int64_t nbl = blocks(nl);
    int64_t nbg = 0;
    uint32_t *kept = nullptr, *sel = nullptr;
    auto count_pass = [&]() -> latentam_status {
        m->epoch += 1;
        nbg = blocks(m->count);
        LAT_TRY(grow_scratch(m, nbl + nbg));
        kept = m->pos, sel = m->pos + nbl;
        if (nl > 0) {
            write_back<<<blocks(nl), kMapThreads, 0, st>>>(nl, local, d, vec_rows(d, local, m->g), m->g, cx, cy, cz,
                                                           r2, m->epoch_mark, m->epoch, kept, m->total + 2);
            LAT_CHECK_LAUNCH("write_back");
        }
        if (m->count > 0) {
            select_global<<<blocks(m->count), kMapThreads, 0, st>>>(m->count, m->g.means, cx, cy, cz, r2,
                                                                    m->epoch_mark, m->epoch, sel);
            LAT_CHECK_LAUNCH("select_global");
        }
        scan_counts<<<2, 1024, 0, st>>>(kept, nbl, sel, nbg, m->total);
        LAT_CHECK_LAUNCH("scan_counts");
        return read_totals(m, 3, st);
    };
    auto insert_new = [&] { return insert_rows(ctx, m, nl, local, local.gidx, nullptr, nullptr, st); };
    auto unstored = [&] { return m->host_total[2] == (uint32_t)m->epoch; };
    const bool first = m->fresh;
    if (first) LAT_TRY(insert_new());
    LAT_TRY(count_pass());
    if (!first && unstored()) {
        LAT_TRY(insert_new());
        LAT_TRY(count_pass());
    }
    m->fresh = unstored();
    const int64_t n_kept = m->host_total[0], n_sel = m->host_total[1], n_new = n_kept + n_sel;
    const int other = m->cur ^ 1;
    LAT_TRY(grow_local(m, other, n_new, 0));
    if (n_kept > 0) {
        compact_local<<<blocks(nl), kMapThreads, 0, st>>>(nl, local, d, vec_rows(d, local, m->loc[other]), cx, cy, cz,
                                                          r2, kept, m->loc[other]);
        LAT_CHECK_LAUNCH("compact_local");
    }
    if (n_sel > 0) {
        append_global<<<blocks(m->count), kMapThreads, 0, st>>>(m->count, m->g, d, vec_rows(d, m->g, m->loc[other]),
                                                                cx, cy, cz, r2, m->epoch_mark, m->epoch, sel,
                                                                (uint32_t)n_sel, n_kept, m->loc[other]);
        LAT_CHECK_LAUNCH("append_global");
    }
    m->cur = other;
    m->local_count = n_new;
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_error(e, "voxel map: sync");
    if (local_out) fill_local(m, local_out);
    return LATENTAM_OK;
}

latentam_status latentam_map_local_view(latentam_map* m, latentam_map_local* out) {
    if (!m || !out) {
        set_error("null map or output");
        return LATENTAM_ERR_INVALID_ARG;
    }
    fill_local(m, out);
    return LATENTAM_OK;
}

latentam_status latentam_map_global_view(latentam_map* m, latentam_map_global* out) {
    if (!m || !out) {
        set_error("null map or output");
        return LATENTAM_ERR_INVALID_ARG;
    }
    *out = latentam_map_global{m->g.means, m->g.quats, m->g.scales, m->g.opac, m->g.f, m->table, m->count,
                               (int64_t)1 << m->table_log2};
    return LATENTAM_OK;
}

}  // extern "C"

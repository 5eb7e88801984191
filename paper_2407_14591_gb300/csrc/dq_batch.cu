// Batched product: y_k = H_k x_k for up to 64 sectors of uneven dimension (different L, N and
// disorder), each with nrhs right-hand sides, in ONE persistent launch.
//
// The rows of all sectors are cut into tiles; tile t belongs to the sector k with
// prefix[k] <= t < prefix[k+1]. CTAs pull tiles from an atomic queue (a counter cleared before
// each launch), copy the descriptor of the tile's sector into shared memory when the sector
// changes, and run the general Q = 2 row computation (bond layers, rank by Eq. (index) or Lin's
// two tables, gather of the columns of x[j], one store of y[i]), a lane per row. The words of a
// warp's rows come from one of two mappings:
//   rows    -- each row unranked with Alg. 4;
//   walk    -- Alg. 4 for a lane's first row of a chunk, then the last subsystem's unrank list.
// The autotuner times every (mapping, threads, CTAs per SM, tile) candidate on the caller's
// vectors and keeps the fastest; a batch with too few rows for two tiles per resident CTA is cut
// into smaller tiles whatever the candidate.
//
// Bound: the FP64 pipe (0.59 T multiply-adds/s) for FP64 vectors, on which every column of every
// hop costs one multiply-add, also for the lanes that wait for a row with more hops. So the
// number of columns is a template argument (no operation for a column that is not there), the
// hops of all bond layers are one sequence, and each warp takes the rows of a 256-row chunk in
// the order of their number of hops. 64 chains of 16 to 26 sites, FP64: 8 columns 26.2 -> 20.2 ms
// (17.9 ms of FP64 operations), 5 columns 22.9 -> 14.0, one column 22.9 -> 6.3; FP32, 8 columns
// 16.7 -> 9.2; six chains of 12 to 16 sites 227 -> 28 us. Without the order 22.3 ms. Lanes that
// share a row (contiguous loads of its columns) repeat the search for the next hop: 28 ms. Two or
// four hops in flight per lane cost registers and with them warps: 25 to 34 ms.
//
// Arithmetic: FP64 vectors accumulate in FP64. FP32 vectors use the FP32 copies of the
// coefficients, form products in FP32 and sum them with Neumaier's compensated summation, so the
// error of each row sum stays at about one FP32 rounding instead of growing with its length.
#include <cstdint>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "dq_device.cuh"
#include "dq_internal.h"

namespace dq {

constexpr int kBatchMax = 64;
constexpr int kBatchMaxRhs = 8;

struct BatchItem {
    DevSector S;
    DevTermsQ2 H;
};

struct BatchParams {
    int n, rows_per_tile, rows_per_warp;
    bool walk;
    unsigned long long total_tiles;
    unsigned long long* queue;      // next tile (cleared before the launch)
    unsigned long long prefix[kBatchMax + 1];  // first tile of each sector
    const BatchItem* items;
    const void* x[kBatchMax];
    void* y[kBatchMax];
};

// Coefficient in the vectors' precision (FP64 vectors: the FP64 value; FP32: its FP32 copy).
template <typename T>
__device__ __forceinline__ T bcf(double d, float f) {
    if constexpr (sizeof(T) == 8)
        return d;
    else
        return f;
}

// V columns of one row in one load (V elements are 4, 8 or 16 bytes; the caller checked the alignment).
template <typename T, int V>
struct alignas(sizeof(T) * V) Cols {
    T v[V];
};
template <typename T, int V>
__device__ __forceinline__ Cols<T, V> load_cols(const T* p) {
    Cols<T, V> r;
    if constexpr (sizeof(T) * V == 16)
        *reinterpret_cast<int4*>(&r) = __ldg(reinterpret_cast<const int4*>(p));
    else if constexpr (sizeof(T) * V == 8)
        *reinterpret_cast<int2*>(&r) = __ldg(reinterpret_cast<const int2*>(p));
    else
        *reinterpret_cast<int*>(&r) = __ldg(reinterpret_cast<const int*>(p));
    return r;
}

// Diagonal of the row with word s: FP64 vectors in FP64; FP32 vectors with FP32 coefficients, compensated.
template <typename T>
__device__ __forceinline__ T batch_diag(const DevTermsQ2& H, uint64_t s) {
    const T* posT = sizeof(T) == 8 ? (const T*)H.pos : (const T*)H.posf;
    const T* linT = sizeof(T) == 8 ? (const T*)H.lin : (const T*)H.linf;
    const T* KT = sizeof(T) == 8 ? (const T*)H.KA : (const T*)H.KAf;
    RowAcc<T> d;
    d.init(bcf<T>(H.C, H.Cf));
    if (linT) {
        uint64_t m = s;
        while (m) {
            const int p = __ffsll((long long)m) - 1;
            m &= m - 1;
            d.add(__ldg(linT + p));
        }
    }
    for (int l = 0; l < H.nl; ++l) {
        uint64_t a = (s ^ (s >> H.dist[l])) & H.dmask[l];
        if (H.kpos[l] < 0) {
            if (a) d.add(__ldg(KT + l) * (T)__popcll(a));
        } else {
            while (a) {
                const int p = __ffsll((long long)a) - 1;
                a &= a - 1;
                d.add(__ldg(posT + H.kpos[l] + p));
            }
        }
    }
    return d.get();
}

constexpr int kSteps = 8;   // 32-row steps of the chunk that a warp orders by hop count
constexpr int kChunk = 32 * kSteps;
constexpr int kBins = 64;

// Shared memory of one warp: the words of its chunk, the order in which it takes them, the hop-count bins.
struct WarpChunk {
    uint64_t word[kChunk];
    int bin[kBins];
    unsigned char order[kChunk];
};
static_assert(kChunk <= 256, "the order holds a byte per row");

// Row i (word s) of sector (S, H): y[i, :] = sum_j H_ij x[j, :] for NR right-hand sides, read V at a time.
template <typename T, int NR, int V>
__device__ __forceinline__ void batch_row(const DevSector& S, const DevTermsQ2& H, const T* __restrict__ x,
                                          T* __restrict__ y, uint64_t i, uint64_t s) {
    const bool lin2 = S.n_sub == 2;
    const T* posT = sizeof(T) == 8 ? (const T*)H.pos : (const T*)H.posf;
    const T* KT = sizeof(T) == 8 ? (const T*)H.KA : (const T*)H.KAf;
    RowAcc<T> acc[NR];
    {
        const T dv = batch_diag<T>(H, s);
#pragma unroll
        for (int c = 0; c < NR; c += V) {
            const Cols<T, V> xv = load_cols<T, V>(x + i * NR + c);
#pragma unroll
            for (int v = 0; v < V; ++v) acc[c + v].init(dv * xv.v[v]);
        }
    }
    // Lin's two tables: a hop inside one half keeps the other half's share of the index
    const uint32_t m1 = lin2 ? (uint32_t)((1ull << (S.nb * S.Lk[1])) - 1) : 0u;
    const int sh0 = S.shift[0];
    const uint64_t* c0_tab = S.c0_tab;
    const uint32_t* rank1 = S.rank_tab[S.tab[lin2 ? 1 : 0]];
    const uint32_t r_own = lin2 ? __ldg(rank1 + ((uint32_t)s & m1)) : 0u;
    const uint64_t c_own = i - r_own;
    // the hops of all layers as one sequence, so that lanes wait for each other once per row and not per layer
    const int nl = H.nl;
    int l = -1, ap = -1;
    uint64_t o = 0, pm = 0;
    T au = (T)0;
    for (;;) {
        while (!o && l + 1 < nl) {
            ++l;
            const int dist = H.dist[l];
            o = (s ^ (s >> dist)) & H.omask[l];
            pm = 1ull | (1ull << dist);
            au = __ldg(KT + kMaxLayers + l);
            ap = H.apos[l];
        }
        if (!o) break;
        const int p = __ffsll((long long)o) - 1;
        o &= o - 1;
        const uint64_t flip = pm << p;
        const uint64_t s2 = s ^ flip;
        uint64_t j;
        if (lin2) {
            const uint64_t c = (flip >> sh0) ? __ldg(c0_tab + (uint32_t)(s2 >> sh0)) : c_own;
            const uint32_t r = ((uint32_t)flip & m1) ? __ldg(rank1 + ((uint32_t)s2 & m1)) : r_own;
            j = checked_rank(S, c + r);
        } else {
            j = d_rank(S, S.off, S.str, s2);
        }
        const T amp = ap >= 0 ? __ldg(posT + ap + p) : au;
        Cols<T, V> xv[NR / V];
#pragma unroll
        for (int c = 0; c < NR / V; ++c) xv[c] = load_cols<T, V>(x + j * NR + c * V);
#pragma unroll
        for (int c = 0; c < NR; ++c) acc[c].add(amp * xv[c / V].v[c % V]);
    }
#pragma unroll
    for (int c = 0; c < NR / V; ++c) {
        Cols<T, V> out;
#pragma unroll
        for (int v = 0; v < V; ++v) out.v[v] = acc[c * V + v].get();
        *reinterpret_cast<Cols<T, V>*>(y + i * NR + c * V) = out;
    }
}

template <typename T, int NR, int V>
__global__ void __launch_bounds__(512, 2) k_batch(BatchParams bp) {
    extern __shared__ __align__(16) unsigned char batch_smem[];
    __shared__ BatchItem it;
    __shared__ unsigned long long s_tile;
    int cur = -1;  // sector whose descriptor is in `it` (same value in every thread)
    const int lane = threadIdx.x & 31;
    WarpChunk& ck = reinterpret_cast<WarpChunk*>(batch_smem)[threadIdx.x >> 5];
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(bp.queue, 1ull);
        __syncthreads();
        const unsigned long long tile = s_tile;
        if (tile >= bp.total_tiles) break;
        int k = 0;
        while (k + 1 < bp.n && bp.prefix[k + 1] <= tile) ++k;
        if (k != cur) {  // uniform across the CTA
            const uint32_t* src = reinterpret_cast<const uint32_t*>(bp.items + k);
            uint32_t* dst = reinterpret_cast<uint32_t*>(&it);
            for (int q = threadIdx.x; q < (int)(sizeof(BatchItem) / 4); q += blockDim.x) dst[q] = src[q];
            __syncthreads();
            cur = k;
        }
        const DevSector& S = it.S;
        const DevTermsQ2& H = it.H;
        const T* x = reinterpret_cast<const T*>(bp.x[k]);
        T* y = reinterpret_cast<T*>(bp.y[k]);
        // the warp's part of the tile, chunk by chunk
        const unsigned long long w0 = (tile - bp.prefix[k]) * (unsigned long long)bp.rows_per_tile +
                                      (unsigned long long)(threadIdx.x >> 5) * bp.rows_per_warp;
        const unsigned long long w1 = min(w0 + (unsigned long long)bp.rows_per_warp, (unsigned long long)S.D);
        for (unsigned long long base = w0; base < w1; base += kChunk) {
            const int rows = (int)min((unsigned long long)kChunk, w1 - base);
            for (int q = lane; q < kBins; q += 32) ck.bin[q] = 0;
            __syncwarp();
            RowWalk<uint64_t> rw;
            unsigned key[kSteps];
#pragma unroll
            for (int r = 0; r < kSteps; ++r) {
                const int q = 32 * r + lane;
                key[r] = 0;
                if (q < rows) {
                    if (bp.walk && r)
                        walk_next(S, S.off, S.str, base + q, rw);
                    else
                        walk_start(S, S.off, S.str, base + q, rw);
                    ck.word[q] = rw.s;
                    int n = 0;
                    for (int l = 0; l < H.nl; ++l) n += __popcll((rw.s ^ (rw.s >> H.dist[l])) & H.omask[l]);
                    key[r] = (unsigned)min(n, kBins - 1);
                    atomicAdd(&ck.bin[key[r]], 1);
                }
            }
            __syncwarp();
            // first position of every bin (two per lane)
            const int b0 = ck.bin[2 * lane], b1 = ck.bin[2 * lane + 1];
            int sum = b0 + b1;
#pragma unroll
            for (int d = 1; d < 32; d *= 2) {
                const int t = __shfl_up_sync(0xffffffffu, sum, d);
                if (lane >= d) sum += t;
            }
            ck.bin[2 * lane] = sum - b0 - b1;
            ck.bin[2 * lane + 1] = sum - b1;
            __syncwarp();
#pragma unroll
            for (int r = 0; r < kSteps; ++r)
                if (32 * r + lane < rows) ck.order[atomicAdd(&ck.bin[key[r]], 1)] = (unsigned char)(32 * r + lane);
            __syncwarp();
            for (int q = lane; q < rows; q += 32) {
                const int at = ck.order[q];
                batch_row<T, NR, V>(S, H, x, y, base + at, ck.word[at]);
            }
            __syncwarp();
        }
        __syncthreads();  // everyone is done with `it` and s_tile before they change
    }
}

// Candidates of the autotuner: (mapping 0 = rows, 1 = walk; threads; CTAs per SM; rows per tile).
struct Shape {
    int walk, threads, per_sm, tile;
};
static const Shape kShapes[] = {{0, 128, 8, 2048}, {0, 256, 4, 4096}, {0, 256, 8, 2048}, {0, 512, 2, 8192},
                                {0, 512, 4, 4096}, {0, 256, 4, 16384}, {1, 128, 8, 1024}, {1, 256, 4, 2048},
                                {1, 256, 8, 1024}, {1, 512, 2, 8192}, {1, 256, 4, 4096}};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);

}  // namespace dq

struct dq_batch {
    int n, nrhs, dtype, shape;
    std::vector<unsigned long long> dims;
    void* items;  // device array of BatchItem, then the tile counter of the work queue
    int device;
};

using namespace dq;

static int batch_launch(dq_batch* b, const void* const* x, void* const* y, cudaStream_t st, int shape) {
    const Shape& sh = kShapes[shape];
    BatchParams bp;
    std::memset(&bp, 0, sizeof bp);
    bp.n = b->n;
    bp.items = reinterpret_cast<const BatchItem*>(b->items);
    bp.queue = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(b->items) + sizeof(BatchItem) * b->n);
    const unsigned long long cap = (unsigned long long)sm_count_cached() * sh.per_sm;
    // a small batch is cut finer, down to 32 rows a warp, so that every resident CTA gets a tile
    int tile = sh.tile;
    unsigned long long t = 0;
    for (;; tile /= 2) {
        t = 0;
        for (int k = 0; k < b->n; ++k) t += (b->dims[k] + tile - 1) / tile;
        if (t >= 2 * cap || tile / 2 < sh.threads) break;
    }
    bp.rows_per_tile = tile;
    bp.rows_per_warp = tile / (sh.threads / 32);
    bp.walk = sh.walk != 0;
    t = 0;
    for (int k = 0; k < b->n; ++k) {
        bp.prefix[k] = t;
        t += (b->dims[k] + tile - 1) / tile;
        bp.x[k] = x[k];
        bp.y[k] = y[k];
    }
    bp.prefix[b->n] = t;
    bp.total_tiles = t;
    const unsigned grid = (unsigned)(t < cap ? (t ? t : 1) : cap);
    const size_t smem = sizeof(WarpChunk) * (sh.threads / 32);
    cudaMemsetAsync(bp.queue, 0, sizeof(unsigned long long), st);
    const int tslot = timing_start(st);
    // Columns per load V: the widest load of at most 16 bytes that divides the row and that every vector is
    // aligned for.
    const int es = b->dtype == DQ_F64 ? 8 : 4;
    int V = 16 / es;
    for (; V > 1; V /= 2) {
        bool ok = b->nrhs % V == 0;
        for (int k = 0; ok && k < b->n; ++k)
            ok = ((reinterpret_cast<uintptr_t>(x[k]) | reinterpret_cast<uintptr_t>(y[k])) % (uintptr_t)(V * es)) == 0;
        if (ok) break;
    }
    bool launched = false;
#define DQ_BATCH(T, nr, v)                                        \
    if (b->nrhs == nr && V == v) {                                \
        k_batch<T, nr, v><<<grid, sh.threads, smem, st>>>(bp);    \
        launched = true;                                          \
    }
#define DQ_BATCH_ALL(T)                                                                            \
    DQ_BATCH(T, 1, 1) DQ_BATCH(T, 2, 1) DQ_BATCH(T, 3, 1) DQ_BATCH(T, 4, 1) DQ_BATCH(T, 5, 1)      \
    DQ_BATCH(T, 6, 1) DQ_BATCH(T, 7, 1) DQ_BATCH(T, 8, 1) DQ_BATCH(T, 2, 2) DQ_BATCH(T, 4, 2)      \
    DQ_BATCH(T, 6, 2) DQ_BATCH(T, 8, 2)
    if (b->dtype == DQ_F64) {
        DQ_BATCH_ALL(double)
    } else {
        DQ_BATCH_ALL(float)
        DQ_BATCH(float, 4, 4) DQ_BATCH(float, 8, 4)
    }
#undef DQ_BATCH_ALL
#undef DQ_BATCH
    if (!launched) return (int)cudaErrorInvalidValue;
    timing_stop(tslot, st, 1);
    return (int)cudaGetLastError();
}

extern "C" {

int dq_batch_make(int n, const dq_sector* const* sectors, const dq_terms* const* terms, int nrhs, int dtype,
                  dq_batch** out) {
    clear_error();
    if (!out || !sectors || !terms) return set_error(DQ_EINVAL, "NULL argument");
    *out = nullptr;
    if (n < 1 || n > kBatchMax) return set_error(DQ_EINVAL, "n must be in [1, %d]", kBatchMax);
    if (nrhs < 1 || nrhs > kBatchMaxRhs) return set_error(DQ_EINVAL, "nrhs must be in [1, %d]", kBatchMaxRhs);
    if (dtype != DQ_F64 && dtype != DQ_F32) return set_error(DQ_EINVAL, "dtype must be DQ_F64 or DQ_F32");
    std::vector<BatchItem> host(n);
    dq_batch* b = new (std::nothrow) dq_batch();
    if (!b) return set_error(DQ_ENOMEM, "host allocation");
    b->n = n;
    b->nrhs = nrhs;
    b->dtype = dtype;
    b->shape = 6;  // the fastest or within 2 % of it on every batch that was timed
    b->items = nullptr;
    for (int k = 0; k < n; ++k) {
        const dq_sector* s = sectors[k];
        const dq_terms* t = terms[k];
        if (!s || !t || t->sector != s) {
            delete b;
            return set_error(DQ_EINVAL, "item %d: NULL or terms of another sector", k);
        }
        if (!s->has_device) {
            delete b;
            return set_error(DQ_ECUDA, "no CUDA device: the sector has host tables only");
        }
        if (!t->q2) {
            delete b;
            return set_error(DQ_EINVAL, "item %d: the batched product serves Q = 2 sectors of one-word states", k);
        }
        host[k].S = s->dev;
        host[k].H = t->q2v;
        b->dims.push_back(s->D);
    }
    cudaError_t e = cudaMalloc(&b->items, sizeof(BatchItem) * n + sizeof(unsigned long long));
    if (e != cudaSuccess) {
        delete b;
        return set_error(DQ_ENOMEM, "cudaMalloc: %s", cudaGetErrorString(e));
    }
    e = cudaMemcpy(b->items, host.data(), sizeof(BatchItem) * n, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(b->items);
        delete b;
        return set_error(DQ_ECUDA, "cudaMemcpy: %s", cudaGetErrorString(e));
    }
    cudaGetDevice(&b->device);
    *out = b;
    return DQ_OK;
}

void dq_batch_free(dq_batch* b) {
    if (!b) return;
    cudaFree(b->items);
    delete b;
}

int dq_batch_matvec(dq_batch* b, const void* const* x, void* const* y, void* stream) {
    clear_error();
    if (!b || !x || !y) return set_error(DQ_EINVAL, "NULL argument");
    for (int k = 0; k < b->n; ++k)
        if (!x[k] || !y[k]) return set_error(DQ_EINVAL, "item %d: NULL vector", k);
    int e = batch_launch(b, x, y, (cudaStream_t)stream, b->shape);
    if (e) return set_error(DQ_ECUDA, "batch launch: %s", cudaGetErrorString((cudaError_t)e));
    return DQ_OK;
}

int dq_batch_shape(dq_batch* b, int shape, int* n_shapes) {
    clear_error();
    if (!b) return set_error(DQ_EINVAL, "NULL argument");
    if (n_shapes) *n_shapes = kNumShapes;
    if (shape < 0) return DQ_OK;
    if (shape >= kNumShapes) return set_error(DQ_EINVAL, "shape must be in [0, %d)", kNumShapes);
    b->shape = shape;
    return DQ_OK;
}

int dq_batch_tune(dq_batch* b, const void* const* x, void* const* y, void* stream, int* choice) {
    clear_error();
    if (!b || !x || !y) return set_error(DQ_EINVAL, "NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    int best_i = b->shape;
    for (int i = 0; i < kNumShapes; ++i) {
        int rc = batch_launch(b, x, y, st, i);  // warm-up
        if (rc) {
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            return set_error(DQ_ECUDA, "batch launch: %s", cudaGetErrorString((cudaError_t)rc));
        }
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) batch_launch(b, x, y, st, i);
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
            best = ms;
            best_i = i;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->shape = best_i;
    if (choice) *choice = best_i;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(DQ_ECUDA, "batch tune: %s", cudaGetErrorString(e));
    return DQ_OK;
}

}  // extern "C"

// Rank and unrank of long lists of states, the sector's tables in shared memory.
//
// The look-ups of Alg. 2 and Alg. 4 go to a different place for every state. Out of L1 such a load is split
// into as many accesses as it has lines; out of shared memory it costs its bank conflicts, three or four
// cycles. Each block therefore copies the offset and stride tables (32 bits an entry when D < 2^32) and the
// local tables (16 bits an entry: a local pattern of at most 16 bits and its local index fit) once and takes
// its share of the list, two states a thread and step.
//
// 2^24 states of 32 sites in three subsystems (35 KB of tables): unrank 262 -> 170 us, rank 410 -> 110 us.
// Bound: integer issue; the list itself, 16 bytes a state, takes 40 us of HBM time.
#include <cstdint>

#include <cuda_runtime.h>

#include "dq_device.cuh"
#include "dq_internal.h"

namespace dq {

constexpr int kThreads = 512;
// Blocks resident per SM: as the registers of the two index widths allow without spills.
constexpr int kBlocks32 = 3, kBlocks64 = 2;
// Tables beyond 64 KB stay with the general kernels: copying 128 KB into every SM costs what the look-ups gain
// (two subsystems of 16 bits, 2^24 states: unrank 173 us there, 189 us here).
constexpr size_t kRankStageMax = 64 * 1024;
// Shorter lists stay there too: at 2^20 states the copies weigh as much as the look-ups (unrank 17 to 25 us
// here and there), at 2^22 it is 54 us here and 72 there (32 sites, three subsystems), 45 and 56 us (14 sites
// with four levels, two subsystems).
constexpr uint64_t kRankLongMin = 1ull << 21;

// Byte offsets inside a block's shared memory.
struct RankStage {
    int str, ss[kMaxTables], tab[kMaxTables], count[kMaxTables];
    int bytes;
};

template <typename I>
__device__ __forceinline__ void stage_tables(const DevSector& S, const RankStage& g, unsigned char* sm, bool inverse) {
    I* off = reinterpret_cast<I*>(sm);
    I* str = reinterpret_cast<I*>(sm + g.str);
    for (int q = threadIdx.x; q < S.os_total; q += kThreads) {
        off[q] = (I)S.off[q];
        str[q] = (I)S.str[q];
    }
    for (int t = 0; t < kMaxTables; ++t) {
        uint16_t* tab = reinterpret_cast<uint16_t*>(sm + g.tab[t]);
        const uint32_t* from = inverse ? S.unrank_tab[t] : S.rank_tab[t];
        for (int q = threadIdx.x; q < g.count[t]; q += kThreads) tab[q] = (uint16_t)from[q];
        if (inverse && g.count[t]) {
            uint32_t* ss = reinterpret_cast<uint32_t*>(sm + g.ss[t]);
            for (int q = threadIdx.x; q < (S.Q - 1) * S.tab_len[t] + 2; q += kThreads) ss[q] = S.sec_start[t][q];
        }
    }
    __syncthreads();
}

template <typename I>
__device__ __forceinline__ I quot(I idx, I st) {
    if constexpr (sizeof(I) == 8) return d_quot(idx, st);
    return idx / st;
}

template <typename I>
__global__ void __launch_bounds__(kThreads, sizeof(I) == 8 ? kBlocks64 : kBlocks32)
    k_state_at_long(DevSector S, RankStage g, const ulonglong2* __restrict__ in, ulonglong2* __restrict__ out,
                    uint64_t n) {
    extern __shared__ __align__(16) unsigned char sm[];
    stage_tables<I>(S, g, sm, true);
    const I* off = reinterpret_cast<const I*>(sm);
    const I* str = reinterpret_cast<const I*>(sm + g.str);
    const int last = S.n_sub - 1;
    for (uint64_t t = blockIdx.x * (uint64_t)kThreads + threadIdx.x; 2 * t < n; t += (uint64_t)gridDim.x * kThreads) {
        const bool two = 2 * t + 1 < n;
        uint64_t raw[2];
        if (two) {
            const ulonglong2 v = __ldg(in + t);
            raw[0] = v.x;
            raw[1] = v.y;
        } else {
            raw[0] = raw[1] = __ldg(reinterpret_cast<const unsigned long long*>(in) + 2 * t);
        }
        I idx[2];
        int lam[2] = {0, 0};
        uint64_t w[2] = {0, 0};
        bool ok[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            ok[e] = raw[e] < S.D;
            idx[e] = ok[e] ? (I)raw[e] : (I)0;
        }
        for (int k = 0; k <= last; ++k) {
            const int tb = S.tab[k], ob = S.os_base[k], ld = S.os_ld[k], nmax = S.nmax[k], sh = S.shift[k];
            const uint16_t* tab = reinterpret_cast<const uint16_t*>(sm + g.tab[tb]);
            const uint32_t* ss = reinterpret_cast<const uint32_t*>(sm + g.ss[tb]);
            int nn[2] = {0, 0};
            I li[2] = {idx[0], idx[1]};  // the last subsystem: offset 0, stride 1
            if (k == last) {
#pragma unroll
                for (int e = 0; e < 2; ++e) nn[e] = S.N - lam[e];
            } else {
                // the largest n with offset(n) <= idx, by halving
                for (int step = 1 << (31 - __clz(nmax)); step; step >>= 1) {
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (nn[e] + step <= nmax && !(idx[e] < off[ob + lam[e] * ld + nn[e] + step])) nn[e] += step;
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int o = ob + lam[e] * ld + nn[e];
                    idx[e] -= off[o];
                    li[e] = quot<I>(idx[e], str[o]);
                    idx[e] -= li[e] * str[o];
                }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                w[e] |= (uint64_t)tab[ss[nn[e]] + (uint32_t)li[e]] << sh;
                lam[e] += nn[e];
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (!ok[e]) {
                w[e] = ~0ull;
                if (e == 0 || two) atomicAdd(S.err, 1);
            }
        if (two)
            out[t] = make_ulonglong2(w[0], w[1]);
        else
            reinterpret_cast<unsigned long long*>(out)[2 * t] = w[0];
    }
}

template <typename I>
__global__ void __launch_bounds__(kThreads, sizeof(I) == 8 ? kBlocks64 : kBlocks32)
    k_index_of_long(DevSector S, RankStage g, const ulonglong2* __restrict__ in, ulonglong2* __restrict__ out,
                    uint64_t n) {
    extern __shared__ __align__(16) unsigned char sm[];
    stage_tables<I>(S, g, sm, false);
    const I* off = reinterpret_cast<const I*>(sm);
    const I* str = reinterpret_cast<const I*>(sm + g.str);
    for (uint64_t t = blockIdx.x * (uint64_t)kThreads + threadIdx.x; 2 * t < n; t += (uint64_t)gridDim.x * kThreads) {
        const bool two = 2 * t + 1 < n;
        uint64_t w[2];
        if (two) {
            const ulonglong2 v = __ldg(in + t);
            w[0] = v.x;
            w[1] = v.y;
        } else {
            w[0] = w[1] = __ldg(reinterpret_cast<const unsigned long long*>(in) + 2 * t);
        }
        bool ok[2];
        I idx[2] = {0, 0};
        int lam[2] = {0, 0};
#pragma unroll
        for (int e = 0; e < 2; ++e) ok[e] = d_valid(S, w[e]);
        for (int k = 0; k < S.n_sub; ++k) {
            const uint16_t* tab = reinterpret_cast<const uint16_t*>(sm + g.tab[S.tab[k]]);
            const int ob = S.os_base[k], ld = S.os_ld[k];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (!ok[e]) continue;
                const uint32_t f = field_of(S, w[e], k);
                const int nn = digit_sum(f, S.nb), o = ob + lam[e] * ld + nn;
                idx[e] += off[o] + str[o] * (I)tab[f];
                lam[e] += nn;
            }
        }
        uint64_t r[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            r[e] = ok[e] ? checked_rank(S, (uint64_t)idx[e]) : ~0ull;
            if (!ok[e] && (e == 0 || two)) atomicAdd(S.err, 1);
        }
        if (two)
            out[t] = make_ulonglong2(r[0], r[1]);
        else
            reinterpret_cast<unsigned long long*>(out)[2 * t] = r[0];
    }
}

static bool stage_layout(const DevSector& S, bool inverse, RankStage& g) {
    const size_t es = S.D >> 32 ? 8 : 4;
    size_t at = (size_t)S.os_total * es;
    g.str = (int)at;
    at += (size_t)S.os_total * es;
    for (int t = 0; t < kMaxTables; ++t) {
        g.ss[t] = g.tab[t] = g.count[t] = 0;
        if (S.tab_len[t] == 0) continue;
        if (S.tab_bits[t] > 16) return false;
        size_t count = (size_t)1 << S.tab_bits[t];  // rank: every pattern; unrank: the valid ones
        if (inverse) {
            count = 1;
            for (int i = 0; i < S.tab_len[t]; ++i) count *= S.Q;
        }
        g.ss[t] = (int)at;
        if (inverse) at += (((size_t)(S.Q - 1) * S.tab_len[t] + 2) * 4 + 7) / 8 * 8;
        g.tab[t] = (int)at;
        g.count[t] = (int)count;
        at += (count * 2 + 7) / 8 * 8;
        if (at > kRankStageMax) return false;
    }
    g.bytes = (int)at;
    return true;
}

// 0: launched; -1: the list is too short, the pointers are not 16-byte aligned or the tables are too large;
// otherwise a CUDA error.
int launch_rank_long(const DevSector& S, bool inverse, const uint64_t* in, uint64_t* out, uint64_t n, cudaStream_t st) {
    RankStage g;
    if (n < kRankLongMin || ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15)) return -1;
    if (!stage_layout(S, inverse, g)) return -1;
    const bool wide = (S.D >> 32) != 0;
    const void* fn = inverse ? (wide ? (const void*)k_state_at_long<uint64_t> : (const void*)k_state_at_long<uint32_t>)
                             : (wide ? (const void*)k_index_of_long<uint64_t> : (const void*)k_index_of_long<uint32_t>);
    if (g.bytes > 40 * 1024)
        if (cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, g.bytes)) return (int)e;
    const uint64_t pairs = (n + 1) / 2;
    const uint64_t need = (pairs + kThreads - 1) / kThreads, cap = (uint64_t)sm_count_cached() * (wide ? kBlocks64 : kBlocks32);
    DevSector s = S;
    const ulonglong2* i2 = reinterpret_cast<const ulonglong2*>(in);
    ulonglong2* o2 = reinterpret_cast<ulonglong2*>(out);
    void* args[] = {&s, &g, &i2, &o2, &n};
    return (int)cudaLaunchKernel(fn, dim3((unsigned)(need < cap ? need : cap)), dim3(kThreads), args, (size_t)g.bytes, st);
}

}  // namespace dq

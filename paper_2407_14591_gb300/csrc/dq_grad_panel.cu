// Coefficient gradients on panels: g_q = sum_i sum_r dy[i, r] (T_q x)[i, r] for Q = 2 and two
// subsystems (P_1 of at most 13 sites, P_0 of at most 16), all terms in one pass over the rows.
//
// With index = c_0(s0) + index_1(s1) the rows of one P_0 pattern are a contiguous panel (dq_panel_pb.cu),
// so a hop needs no rank per row: inside P_0 it pairs dy with another panel element by element, inside
// P_1 and across the cut with an element of the panel or of the panel s0 ^ bit_a through a rank table in
// shared memory. Per panel and hop pair each thread sums its rows' dy * x in 64-bit integers (x and dy
// split in 32-bit halves), rounds the sum once onto a common grid 2^-G and a warp adds it to its own
// accumulator. The diagonal terms need only p_i = dy_i x_i, rounded one by one: its sum per panel (P_0
// terms), per P_1 pattern (P_1 terms), and per panel and P_1 bit (pairs across the cut); a last kernel
// forms every term from those. All sums are integers, so the result does not depend on the order of the
// blocks. A block empties its accumulators into the two-word totals before one of them can fill, so the
// grid keeps 48 bits, shared out over the columns, for any number of panels and columns.
//
// Before (one term after the other per row, every hop ranked, 32 terms per launch): 72 terms of the
// 24-site disordered chain (2.7 M rows) 1.0 ms in three launches plus 72 us of final sums. Now 167 us
// (k_grad_panel) and 21 us (k_grad_terms), the scaling of x and dy 29 us; the differentiable step around
// it 1.70 -> 0.76 ms. Bound: integer issue, as for the product.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <map>
#include <vector>

#include <cuda_runtime.h>

#include "dq_fixed.cuh"
#include "dq_grad.h"
#include "dq_internal.h"

namespace dq {

constexpr int kGPT = 256;        // threads per CTA
constexpr int kGPW = kGPT / 32;
constexpr int kGPSlots = 2;      // cut partner panels held at a time
constexpr int kGPPairs = 64;     // hop pairs of one place (P_0, P_1, cut); pairs of the cut with a diagonal
constexpr int kGPGroups = 16;
constexpr int kGPBits = 48;      // |dy x| on the grid, summed over the columns
// rows of one column that a warp or a P_1 pattern may add up before its sum is emptied: below 2^62
constexpr uint64_t kGPRows = 1ull << (62 - kGPBits);

struct GradPlan {
    int L0, L1, N, cap, npair;
    uint32_t npanels;
    const uint32_t* s0;      // P_0 patterns in canonical order, from the first valid one
    const uint64_t* c0;      // first index of every P_0 pattern's panel
    const uint32_t* rank1;   // local index of every P_1 pattern
    const uint32_t* states;  // P_1 patterns grouped by particle number
    uint32_t t1start[15], t1len[15];
    // hop pairs: accumulator k of P_0 pair k, then n0 + k of P_1 pair k, then n0 + n1 + k of the cut's
    int n0, n1, nx;
    uint32_t p0mask[kGPPairs];
    uint32_t p1_lo2[kGPPairs], p1_pm2[kGPPairs];  // shifted left by one (byte offsets into the rank table)
    int p1_d[kGPPairs];
    int nxg, xg_first[kGPGroups + 1];             // cut pairs grouped by their P_0 bit
    uint32_t xg_abit[kGPGroups], xb_bit2[kGPPairs];
    // diagonal pairs across the cut: accumulator n0 + n1 + nx + k holds the sum of p over s_a != s_b;
    // grouped by the P_1 bit
    int nzb, zb_first[16], zb_bit[16];
    uint32_t za[kGPPairs];
};

// One output: f * (sum over the source of sign(kind, bits) p), see k_grad_terms.
struct GradOut {
    int type, kind;       // type: 0 hop accumulator, 1 P_0 patterns, 2 P_1 patterns, 3 pair across the cut
    int i, j;             // bit positions in s0 / s1 (type 3: i in s0, j in s1); type 0: the accumulator
    int acc;              // type 3: accumulator of the pair
};

// Where a call's integers are collected (zeroed before): sums per panel; per P_1 pattern and per
// accumulator as low 32 bits and the rest, so that no total overflows.
struct GradSums {
    unsigned long long *V, *Wlo, *Whi, *Alo, *Ahi;
};

__device__ __forceinline__ void grad_red(unsigned long long* lo, unsigned long long* hi, long long v) {
    atomicAdd(lo, (unsigned long long)(v & 0xffffffffll));
    atomicAdd(hi, (unsigned long long)(v >> 32));
}

// (hh 2^56 + mid 2^28 + ll) 2^-sh, rounded to nearest on the way to units of 2^56 (28 bits below them
// kept, so ties do not bias the sum) and to even on the grid; 64 <= sh.
__device__ __forceinline__ long long grad_grid(const Acc3& a, int sh) {
    const int k = sh - 56;
    if (k > 62) return 0;
    const long long t = a.hh + ((a.mid + (a.ll >> 28) + (1ll << 27)) >> 28);
    return (t + ((1ll << (k - 1)) - 1) + ((t >> k) & 1)) >> k;
}

__device__ __forceinline__ void grad_mac(Acc3& a, long long x, long long y) {
    acc_hop(a, make_int2((int)(x >> 32), (int)x), y);
}

__device__ __forceinline__ long long grad_warp(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Shared memory: the P_1 rank table (u16 byte offsets, one entry more that points at a zero element),
// the panel's x and kGPSlots cut partners (cap + 8 elements each), the sums per P_1 pattern, the warps'
// accumulators.
struct GradSmem {
    int own, bstride, W, acc, total;
    __host__ __device__ GradSmem(const GradPlan& P) {
        auto al = [](int b) { return (b + 127) & ~127; };
        own = al((1 << P.L1) * 2 + 16);
        bstride = al((P.cap + 8) * 8);
        W = own + (1 + (P.nxg ? kGPSlots : 0)) * bstride;
        acc = W + (8 << P.L1);
        total = acc + kGPW * P.npair * 8;
    }
};

__device__ __forceinline__ void grad_copy(long long* dst, const long long* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// The rows of one panel and column, tid + e * kGPT (e < E).
template <int E>
__device__ __forceinline__ void grad_rows(const GradPlan& P, const GradSmem& L, unsigned char* smem,
                                          const long long* __restrict__ X, const long long* __restrict__ DY,
                                          uint32_t s0, uint64_t start, int n1, int C, int sh, unsigned long long* V) {
    const int tid = threadIdx.x, lane = tid & 31;
    unsigned char* own = smem + L.own;
    long long* acc = reinterpret_cast<long long*>(smem + L.acc) + (tid >> 5) * P.npair;
    const uint32_t* states = P.states + P.t1start[n1];
    uint32_t s2[E];
    long long dy[E];  // zero past the panel: such rows add nothing
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = tid + e * kGPT;
        s2[e] = c < C ? __ldg(states + c) << 1 : 0u;
        dy[e] = c < C ? __ldg(DY + start + c) : 0;
    }
    auto finish = [&](int k, const Acc3& a) {
        const long long v = grad_warp(grad_grid(a, sh));
        if (lane == 0) acc[k] += v;
    };
    // hop pairs inside P_0, while the copies of the panel and of the first cut partners land
    // (the next partner's loads are in flight behind the current one's products)
    auto active = [&](int k) {
        while (k < P.n0 && __popc(s0 & P.p0mask[k]) != 1) ++k;
        return k;
    };
    auto load = [&](int k, long long* v) {
        const long long* src = X + __ldg(P.c0 + (s0 ^ P.p0mask[k]));
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = tid + e * kGPT < C ? __ldg(src + tid + e * kGPT) : 0;
    };
    long long v0[E], v1[E];
    int k0 = active(0);
    if (k0 < P.n0) load(k0, v0);
    while (k0 < P.n0) {
        const int k1 = active(k0 + 1);
        if (k1 < P.n0) load(k1, v1);
        Acc3 a = {0, 0, 0};
#pragma unroll
        for (int e = 0; e < E; ++e) grad_mac(a, dy[e], v0[e]);
        finish(k0, a);
#pragma unroll
        for (int e = 0; e < E; ++e) v0[e] = v1[e];
        k0 = k1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    auto at = [&](const unsigned char* base, uint32_t t) {
        return *reinterpret_cast<const long long*>(base + *reinterpret_cast<const uint16_t*>(smem + t));
    };
    const uint32_t zslot = 2u << P.L1;
    // diagonal: p_i per P_1 pattern, per panel, per panel and bit
    long long p[E], all = 0;
    long long* W = reinterpret_cast<long long*>(smem + L.W) + P.t1start[n1];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = tid + e * kGPT;
        p[e] = 0;
        if (c < C) {
            Acc3 a = {0, 0, 0};
            grad_mac(a, dy[e], reinterpret_cast<const long long*>(own)[c]);
            p[e] = grad_grid(a, sh);
            W[c] += p[e];
            all += p[e];
        }
    }
    all = grad_warp(all);
    if (lane == 0) atomicAdd(V, (unsigned long long)all);
    for (int z = 0; z < P.nzb; ++z) {
        long long v = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) v += (s2[e] >> (P.zb_bit[z] + 1)) & 1u ? p[e] : 0;
        v = grad_warp(v);
        if (lane == 0)
            for (int k = P.zb_first[z]; k < P.zb_first[z + 1]; ++k)
                acc[P.n0 + P.n1 + P.nx + k] += (s0 & P.za[k]) ? all - v : v;
    }
    // hop pairs inside P_1
    for (int k = 0; k < P.n1; ++k) {
        const uint32_t lo2 = P.p1_lo2[k], pm2 = P.p1_pm2[k];
        const int d = P.p1_d[k];
        Acc3 a = {0, 0, 0};
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t t = ((s2[e] ^ (s2[e] >> d)) & lo2) ? s2[e] ^ pm2 : zslot;
            grad_mac(a, dy[e], at(own, t));
        }
        finish(P.n0 + k, a);
    }
    // hop pairs across the cut
    for (int g0 = 0; g0 < P.nxg; g0 += kGPSlots) {
        if (g0) {
            __syncthreads();
            for (int j = 0; j < kGPSlots && g0 + j < P.nxg; ++j) {
                const int np = (s0 & P.xg_abit[g0 + j]) ? n1 + 1 : n1 - 1;
                if (np < 0 || np > P.L1) continue;
                const long long* src = X + __ldg(P.c0 + (s0 ^ P.xg_abit[g0 + j]));
                long long* dst = reinterpret_cast<long long*>(own + (1 + j) * L.bstride);
                for (int c = tid; c < (int)P.t1len[np]; c += kGPT) grad_copy(dst + c, src + c);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
        }
        for (int j = 0; j < kGPSlots && g0 + j < P.nxg; ++j) {
            const int g = g0 + j;
            const bool sa = (s0 & P.xg_abit[g]) != 0;
            const int np = sa ? n1 + 1 : n1 - 1;
            if (np < 0 || np > P.L1) continue;  // no partner: no row of the panel hops here
            const unsigned char* slot = own + (1 + j) * L.bstride;
            for (int k = P.xg_first[g]; k < P.xg_first[g + 1]; ++k) {
                const uint32_t bb2 = P.xb_bit2[k], flip = sa ? ~0u : 0u;
                Acc3 a = {0, 0, 0};
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint32_t t = ((s2[e] ^ flip) & bb2) ? s2[e] ^ bb2 : zslot;
                    grad_mac(a, dy[e], at(slot, t));
                }
                finish(P.n0 + P.n1 + k, a);
            }
        }
    }
}

__device__ __forceinline__ void grad_scales(const ColScale* hx, const ColScale* hdy, int cols, int* G, int* sh) {
    // common grid: the largest column bound of |dy x| lands below 2^(kGPBits - lg cols)
    int lg = 0;
    while ((1 << lg) < cols) ++lg;
    int fmin = 1 << 30;
    for (int r = 0; r < cols; ++r) fmin = min(fmin, hx->F[r] + hdy->F[r]);
    *G = fmin - (112 - kGPBits) - lg;  // |X| and |DY| stay below 2^56
    for (int r = 0; sh && r < cols; ++r) sh[r] = hx->F[r] + hdy->F[r] - *G;
}

__global__ void __launch_bounds__(kGPT, 2)
    k_grad_panel(GradPlan P, GradSmem L, const long long* __restrict__ X, const long long* __restrict__ DY,
                 const ColScale* __restrict__ hx, const ColScale* __restrict__ hdy, uint64_t xstride, int cols, int period,
                 GradSums out) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int sh_s[kMaxCols], G_s;
    const int tid = threadIdx.x;
    if (hx->bad | hdy->bad) return;  // the last kernel reports it
    uint16_t* t1 = reinterpret_cast<uint16_t*>(smem);
    const uint32_t ntab = 1u << P.L1;
    for (uint32_t q = tid; q <= ntab; q += kGPT)
        t1[q] = (uint16_t)((q < ntab ? __ldg(P.rank1 + q) : (uint32_t)P.cap) * 8);
    for (int q = tid; q < 8 * (1 + (P.nxg ? kGPSlots : 0)); q += kGPT)
        reinterpret_cast<long long*>(smem + L.own + (q / 8) * L.bstride)[P.cap + q % 8] = 0;
    for (uint32_t q = tid; q < ntab; q += kGPT) reinterpret_cast<long long*>(smem + L.W)[q] = 0;
    for (int q = tid; q < kGPW * P.npair; q += kGPT) reinterpret_cast<long long*>(smem + L.acc)[q] = 0;
    if (tid == 0) grad_scales(hx, hdy, cols, &G_s, sh_s);
    // the block's sums into the totals, and from zero again (between two barriers)
    auto empty = [&]() {
        for (uint32_t q = tid; q < ntab; q += kGPT) {
            long long& v = reinterpret_cast<long long*>(smem + L.W)[q];
            if (v) grad_red(out.Wlo + q, out.Whi + q, v);
            v = 0;
        }
        for (int q = tid; q < P.npair; q += kGPT) {
            long long hi = 0;  // a warp's sums stay below 2^62, eight of them below 2^65
            unsigned long long lo = 0;
            for (int w = 0; w < kGPW; ++w) {
                long long& a = reinterpret_cast<long long*>(smem + L.acc)[w * P.npair + q];
                lo += (unsigned long long)(a & 0xffffffffll);
                hi += a >> 32;
                a = 0;
            }
            atomicAdd(out.Alo + q, lo);
            atomicAdd(out.Ahi + q, (unsigned long long)hi);
        }
    };
    const uint64_t items = (uint64_t)P.npanels * cols;
    int since = 0;  // items since the sums were last emptied
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const uint32_t pi = (uint32_t)(item / cols);
        const int col = (int)(item % cols);
        const uint32_t s0 = __ldg(P.s0 + pi);
        const uint64_t start = __ldg(P.c0 + s0);
        const int n1 = P.N - __popc(s0), C = (int)P.t1len[n1];
        const long long* Xc = X + col * xstride;
        __syncthreads();  // the previous panel is finished
        if (since == period) {
            empty();
            __syncthreads();  // a warp's own rows begin with its accumulators
            since = 0;
        }
        ++since;
        long long* own = reinterpret_cast<long long*>(smem + L.own);
        for (int c = tid; c < C; c += kGPT) grad_copy(own + c, Xc + start + c);
        for (int j = 0; j < kGPSlots && j < P.nxg; ++j) {
            const int np = (s0 & P.xg_abit[j]) ? n1 + 1 : n1 - 1;
            if (np < 0 || np > P.L1) continue;
            const long long* src = Xc + __ldg(P.c0 + (s0 ^ P.xg_abit[j]));
            long long* dst = reinterpret_cast<long long*>(smem + L.own + (1 + j) * L.bstride);
            for (int c = tid; c < (int)P.t1len[np]; c += kGPT) grad_copy(dst + c, src + c);
        }
        const int sh = sh_s[col];
#define GRAD_ROWS(e) grad_rows<e>(P, L, smem, Xc, DY + col * xstride, s0, start, n1, C, sh, out.V + pi)
        switch ((C + kGPT - 1) / kGPT) {
            case 7: GRAD_ROWS(7); break;
            case 6: GRAD_ROWS(6); break;
            case 5: GRAD_ROWS(5); break;
            case 4: GRAD_ROWS(4); break;
            case 3: GRAD_ROWS(3); break;
            case 2: GRAD_ROWS(2); break;
            default: GRAD_ROWS(1);
        }
#undef GRAD_ROWS
    }
    __syncthreads();
    empty();
}

// Output q, one block each: f * sum of sign * p in units of 2^-G.
__global__ void __launch_bounds__(256)
    k_grad_terms(GradPlan P, GradSums in, const GradOut* __restrict__ outs, const ColScale* __restrict__ hx,
                 const ColScale* __restrict__ hdy, int cols, double* __restrict__ g, int* err) {
    __shared__ long long red[2][8];
    const GradOut o = outs[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31;
    // sums of twice (type 3) or once the sign times p, split as lo + hi 2^32
    long long lo = 0, hi = 0;
    auto sign = [&](int ni, int nj) -> int {
        switch (o.kind) {
            case DQ_ZZ: return ni == nj ? 1 : -1;
            case DQ_Z: return ni ? 1 : -1;
            case DQ_NN: return ni & nj;
            case DQ_N: return ni;
            default: return 0;  // DQ_U: n (n - 1) = 0 for Q = 2
        }
    };
    auto add = [&](unsigned long long l, unsigned long long h, int m) {
        lo += m * (long long)l;
        hi += m * (long long)h;
    };
    if (o.type == 1 || o.type == 3)
        for (uint32_t q = tid; q < P.npanels; q += 256) {
            const uint32_t s = __ldg(P.s0 + q);
            const long long v = (long long)__ldcg(in.V + q);
            // type 3: ZZ = sum - 2 D, NN = (N_i + N_j - D) / 2
            const int m = o.type == 1 ? sign((s >> o.i) & 1u, (s >> o.j) & 1u) : o.kind == DQ_ZZ ? 1 : (int)((s >> o.i) & 1u);
            add((unsigned long long)(v & 0xffffffffll), (unsigned long long)(v >> 32), m);
        }
    if (o.type == 2 || (o.type == 3 && o.kind == DQ_NN))
        for (uint32_t q = tid; q < (1u << P.L1); q += 256) {
            const uint32_t s = __ldg(P.states + q);
            const int m = o.type == 2 ? sign((s >> o.i) & 1u, (s >> o.j) & 1u) : (int)((s >> o.j) & 1u);
            add(__ldcg(in.Wlo + q), __ldcg(in.Whi + q), m);
        }
    if (tid == 0 && (o.type == 0 || o.type == 3))
        add(__ldcg(in.Alo + o.acc), __ldcg(in.Ahi + o.acc), o.type == 0 ? 1 : o.kind == DQ_ZZ ? -2 : -1);
    lo = grad_warp(lo);
    hi = grad_warp(hi);
    if (lane == 0) {
        red[0][tid >> 5] = lo;
        red[1][tid >> 5] = hi;
    }
    __syncthreads();
    if (tid == 0) {
        lo = hi = 0;
        for (int w = 0; w < 8; ++w) {
            lo += red[0][w];
            hi += red[1][w];
        }
        hi += lo >> 32;
        lo &= 0xffffffffll;
        double f = 1.0;
        switch (o.kind) {
            case DQ_ZZ: f = 0.25; break;
            case DQ_Z: f = 0.5; break;
            case DQ_XY: f = 0.5; break;
            case DQ_HOP: f = -1.0; break;
            case DQ_NN: f = o.type == 3 ? 0.5 : 1.0; break;
            default: break;
        }
        int G;
        if (hx->bad | hdy->bad) {  // an Inf or NaN in x or dy
            g[blockIdx.x] = __longlong_as_double(0x7ff8000000000000ll);
            if (blockIdx.x == 0) atomicAdd(err, 1);
        } else {
            grad_scales(hx, hdy, cols, &G, nullptr);
            g[blockIdx.x] = ldexp(f * ((double)hi * 4294967296.0 + (double)lo), -G);
        }
    }
}

// Largest exponents of the columns of x (blockIdx.y = 0) and dy (1).
template <typename T>
__global__ void k_grad_exp_max(const T* __restrict__ x, const T* __restrict__ dy, uint64_t n, int ld, ColScale* hx, ColScale* hdy) {
    using U = typename FBits<T>::U;
    __shared__ int m_s[kMaxCols];
    const U* v = reinterpret_cast<const U*>(blockIdx.y ? dy : x);
    ColScale* h = blockIdx.y ? hdy : hx;
    for (int c = threadIdx.x; c < ld; c += blockDim.x) m_s[c] = 0;
    __syncthreads();
    const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
    int m = 0;
#pragma unroll 4
    for (uint64_t i = t0; i < n; i += step) m = max(m, exp_field<T>(__ldg(v + i)));
    if (m) atomicMax(&m_s[(int)(t0 % (uint64_t)ld)], m);
    __syncthreads();
    for (int c = threadIdx.x; c < ld; c += blockDim.x)
        if (m_s[c]) atomicMax(&h->emax[c], m_s[c]);
}

// The columns of x (blockIdx.y = 0) and dy (1) as split words, xstride elements apart.
template <typename T>
__global__ void k_grad_fixed(const T* __restrict__ x, const T* __restrict__ dy, long long* __restrict__ X,
                             long long* __restrict__ DY, uint64_t n, int cols, uint64_t xstride, ColScale* hx, ColScale* hdy) {
    using U = typename FBits<T>::U;
    const U* v = reinterpret_cast<const U*>(blockIdx.y ? dy : x);
    long long* to = blockIdx.y ? DY : X;
    ColScale* h = blockIdx.y ? hdy : hx;
    const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
    const int c = (int)(t0 % (uint64_t)cols);
    const int emax = h->emax[c];
    const int F = XHead<long long>::HEAD - (emax - FBits<T>::BIAS + 1);
    if (t0 < (uint64_t)cols) {
        h->F[c] = F;
        if (emax == FBits<T>::EMASK) h->bad = 1;
    }
    if (emax == FBits<T>::EMASK) return;
#pragma unroll 4
    for (uint64_t i = t0; i < n; i += step)
        to[cols == 1 ? i : c * xstride + i / cols] = split_word(to_fixed<T, long long>(__ldg(v + i), F));
}

// ------------------------------------------------------------------ host --------------------

// Where the pass over panels pays. It works on the columns one after the other, the general kernels rank a
// hop once for all columns; it shares a panel's loads among all terms; and its frame around a panel is the
// same for a short one. With one column it is always the faster. Measured, us, general against panels, by
// rows a panel:
//   little work, bound by launches: 20 sites, N = 6 (46 rows), four columns 297 / 216; N = 10 (180), eight
//     413 / 345, sixteen and eight terms 251 / 245; 24 sites, N = 6 (54), two 416 / 299, three and 24 terms 194 / 235;
//   few terms: 24 sites, N = 12 (660 rows), eight terms and four columns 432 / 387, eight columns 640 / 680;
//     N = 9 (325) two 239 / 187, four 283 / 304; 26 sites, N = 6 (56) two 168 / 154 but 78 terms 453 / 602;
//   many terms: 24 sites, N = 12, 72 terms, eight columns 4164 / 1648, 24 terms and sixteen 3588 / 2490; N = 9,
//     72 terms and sixteen 3762 / 2602, eight terms 794 / 1082; 26 sites, N = 9 (400), 78 terms and sixteen 8999 /
//     9201; 22 sites, N = 11 (344), 66 terms and 32 3551 / 2967, eight terms 881 / 1525.
static bool grad_pays(uint64_t D, uint32_t npanels, int n_terms, int cols) {
    const uint64_t rows = D / npanels, items = (uint64_t)npanels * cols;
    return cols == 1 || items <= (rows >= 150 ? 8192 : 5120) || (cols <= 4 && rows >= 160 * (uint64_t)cols) ||
           (cols <= 16 && rows >= 300 && (uint64_t)n_terms * rows >= 9600);
}

// The plan for a term list; false when it does not fit (too many pairs of one place, or the sector) or
// would not pay.
static bool grad_plan(const dq_sector* s, const dq_term* terms, int n_terms, int cols, GradPlan& P, std::vector<GradOut>& outs) {
    if (s->Q != 2 || s->n_sub != 2 || s->wide) return false;
    const int L = s->L, L0 = s->Lk[0], L1 = s->Lk[1], N = s->N;
    if (L1 < 1 || L1 > 13 || L0 > 16) return false;
    std::memset(&P, 0, sizeof P);
    P.L0 = L0;
    P.L1 = L1;
    P.N = N;
    const auto& s0s = s->h.sec_start[s->dev.tab[0]];
    const auto& s1s = s->h.sec_start[s->dev.tab[1]];
    const int a = std::max(0, N - L1), b = std::min(L0, N);  // particle numbers of P_0
    P.s0 = s->dev.unrank_tab[s->dev.tab[0]] + s0s[a];
    P.npanels = s0s[b + 1] - s0s[a];
    if (!grad_pays(s->D, P.npanels, n_terms, cols)) return false;
    P.c0 = s->dev.c0_tab;
    P.rank1 = s->dev.rank_tab[s->dev.tab[1]];
    P.states = s->dev.unrank_tab[s->dev.tab[1]];
    for (int n = 0; n <= L1; ++n) {
        P.t1start[n] = s1s[n];
        P.t1len[n] = s1s[n + 1] - s1s[n];
        if (N - n >= 0 && N - n <= L0) P.cap = std::max(P.cap, (int)P.t1len[n]);
    }
    // distinct hop pairs and diagonal pairs across the cut, by place
    std::map<std::pair<int, int>, int> h0, h1, hx, zx;  // (hi, lo) bits -> index (hx, zx: by group below)
    outs.resize(n_terms);
    for (int q = 0; q < n_terms; ++q) {
        const dq_term& u = terms[q];
        GradOut& o = outs[q];
        std::memset(&o, 0, sizeof o);
        o.kind = u.kind;
        const bool pair = u.kind == DQ_XY || u.kind == DQ_ZZ || u.kind == DQ_HOP || u.kind == DQ_NN;
        const bool hop = u.kind == DQ_XY || u.kind == DQ_HOP;
        const int pi = L - 1 - u.i, pj = pair ? L - 1 - u.j : pi, hi = std::max(pi, pj), lo = std::min(pi, pj);
        if (lo >= L1) {
            o.type = 1;
            o.i = hi - L1;
            o.j = lo - L1;
            if (hop) h0.emplace(std::make_pair(hi, lo), 0);
        } else if (hi < L1) {
            o.type = 2;
            o.i = hi;
            o.j = lo;
            if (hop) h1.emplace(std::make_pair(hi, lo), 0);
        } else {
            o.type = 3;
            o.i = hi - L1;
            o.j = lo;
            if (hop)
                hx.emplace(std::make_pair(hi, lo), 0);
            else
                zx.emplace(std::make_pair(lo, hi), 0);
        }
    }
    if (h0.size() > (size_t)kGPPairs || h1.size() > (size_t)kGPPairs || hx.size() > (size_t)kGPPairs ||
        zx.size() > (size_t)kGPPairs)
        return false;
    for (auto& e : h0) {
        e.second = P.n0;
        P.p0mask[P.n0++] = (1u << (e.first.first - L1)) | (1u << (e.first.second - L1));
    }
    for (auto& e : h1) {
        e.second = P.n0 + P.n1;
        P.p1_lo2[P.n1] = 2u << e.first.second;
        P.p1_d[P.n1] = e.first.first - e.first.second;
        P.p1_pm2[P.n1++] = (2u << e.first.first) | (2u << e.first.second);
    }
    int last = -1;
    for (auto& e : hx) {  // ordered by the P_0 bit
        if (e.first.first != last) {
            last = e.first.first;
            P.xg_abit[P.nxg] = 1u << (last - L1);
            P.xg_first[P.nxg++] = P.nx;
        }
        e.second = P.n0 + P.n1 + P.nx;
        P.xb_bit2[P.nx++] = 2u << e.first.second;
    }
    P.xg_first[P.nxg] = P.nx;
    int nz = 0;
    last = -1;
    for (auto& e : zx) {  // ordered by the P_1 bit
        if (e.first.first != last) {
            last = e.first.first;
            P.zb_bit[P.nzb] = last;
            P.zb_first[P.nzb++] = nz;
        }
        e.second = P.n0 + P.n1 + P.nx + nz;
        P.za[nz++] = 1u << (e.first.second - L1);
    }
    P.zb_first[P.nzb] = nz;
    P.npair = P.n0 + P.n1 + P.nx + nz;
    for (int q = 0; q < n_terms; ++q) {
        GradOut& o = outs[q];
        const bool hop = o.kind == DQ_XY || o.kind == DQ_HOP;
        if (hop) {
            o.acc = o.type == 1 ? h0[{o.i + L1, o.j + L1}] : o.type == 2 ? h1[{o.i, o.j}] : hx[{o.i + L1, o.j}];
            o.type = 0;
        } else if (o.type == 3) {
            o.acc = zx[{o.j, o.i + L1}];
        }
    }
    return true;
}

int launch_grad_panel(const dq_sector* s, const dq_term* terms, int n_terms, const void* x, const void* dy, int dtype,
                      int cols, double* d_grads, cudaStream_t st, bool* taken) {
    GradPlan P;
    std::vector<GradOut> outs;
    *taken = grad_plan(s, terms, n_terms, cols, P, outs);
    if (!*taken) return 0;
    const GradSmem L(P);
    const int sms = sm_count_cached();
    auto kern = k_grad_panel;
    if (L.total > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L.total);
        if (e != cudaSuccess) return (int)e;
    }
    const int per_sm = occupancy_cached(reinterpret_cast<const void*>(kern), kGPT, L.total);
    const uint64_t items = (uint64_t)P.npanels * cols;
    const unsigned grid = (unsigned)std::min<uint64_t>(std::max<uint64_t>(items, 1), (uint64_t)sms * per_sm);
    // items of a block between two emptyings: a warp takes up to this many rows of a panel
    const uint64_t rows = (uint64_t)((P.cap + kGPT - 1) / kGPT) * 32;
    const int period = (int)(kGPRows / rows);
    // workspace: the two scales and the sums (zeroed), the outputs, the copies of x and dy
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const uint64_t xstride = (s->D + 15) & ~15ull;
    const size_t o_v = 2 * kColScaleBytes, o_w = o_v + al(8 * (size_t)P.npanels), o_a = o_w + ((size_t)16 << P.L1);
    const size_t o_out = o_a + al(16 * (size_t)std::max(1, P.npair)), o_x = o_out + al(sizeof(GradOut) * outs.size());
    const size_t vec = al(xstride * cols * 8), need = o_x + 2 * vec;
    char* ws = nullptr;
    if (int rc = grad_workspace(s, need, &ws)) return rc;
    ColScale* hx = reinterpret_cast<ColScale*>(ws);
    ColScale* hdy = reinterpret_cast<ColScale*>(ws + kColScaleBytes);
    GradSums sum;
    sum.V = reinterpret_cast<unsigned long long*>(ws + o_v);
    sum.Wlo = reinterpret_cast<unsigned long long*>(ws + o_w);
    sum.Whi = sum.Wlo + ((size_t)1 << P.L1);
    sum.Alo = reinterpret_cast<unsigned long long*>(ws + o_a);
    sum.Ahi = sum.Alo + std::max(1, P.npair);
    GradOut* d_out = reinterpret_cast<GradOut*>(ws + o_out);
    long long* X = reinterpret_cast<long long*>(ws + o_x);
    long long* DY = reinterpret_cast<long long*>(ws + o_x + vec);
    cudaMemsetAsync(ws, 0, o_out, st);
    cudaError_t e = cudaMemcpyAsync(d_out, outs.data(), sizeof(GradOut) * outs.size(), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return (int)e;
    const int tslot = timing_start(st);
    const int bs = col_block(cols);
    const uint64_t n = s->D * (uint64_t)cols;
    const dim3 pgrid((unsigned)std::min<uint64_t>((n + bs - 1) / bs, (uint64_t)sms * 4), 2);
    if (dtype == DQ_F64) {
        k_grad_exp_max<double><<<pgrid, bs, 0, st>>>((const double*)x, (const double*)dy, n, cols, hx, hdy);
        k_grad_fixed<double><<<pgrid, bs, 0, st>>>((const double*)x, (const double*)dy, X, DY, n, cols, xstride, hx, hdy);
    } else {
        k_grad_exp_max<float><<<pgrid, bs, 0, st>>>((const float*)x, (const float*)dy, n, cols, hx, hdy);
        k_grad_fixed<float><<<pgrid, bs, 0, st>>>((const float*)x, (const float*)dy, X, DY, n, cols, xstride, hx, hdy);
    }
    kern<<<grid, kGPT, L.total, st>>>(P, L, X, DY, hx, hdy, xstride, cols, period, sum);
    k_grad_terms<<<n_terms, 256, 0, st>>>(P, sum, d_out, hx, hdy, cols, d_grads, s->dev.err);
    timing_stop(tslot, st, 4);
    return (int)cudaGetLastError();
}

}  // namespace dq

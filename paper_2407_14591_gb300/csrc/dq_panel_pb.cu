// Per-bond panel product: the structural rank of the panel product (dq_panel.cu) for operators
// whose couplings and fields differ from bond to bond and from site to site (disordered chains
// and lattices), Q = 2, two subsystems, P_1 of at most 13 sites.
//
// With index = c_0(s0) + index_1(s1) (Sec. 3.3, Lin's two tables) the rows sharing a P_0 pattern
// s0 form a contiguous panel of C(L_1, n_1) rows. Per panel (one CTA of 256 threads, three per SM):
//   - the panel's x (fixed point, from the one-column prepass) and up to four partner panels across the
//     cut are copied into shared memory asynchronously, next to the P_1 rank table (byte offsets of the
//     local index of every P_1 pattern);
//   - meanwhile the hops inside P_0 read their partner panels element by element (coalesced, several
//     partners in flight);
//   - hops inside P_1 are gathers through the rank table; a pair whose bits are equal reads an element
//     that holds zero, so the lanes never branch;
//   - hops across the cut gather from the partner panels s0 ^ bit_a the same way;
//   - the diagonal is a table value per P_1 pattern (its fields and Sz Sz bonds) plus two sums per panel
//     in shared memory (the panel's constant and the cut bonds by the low and the high P_1 bits).
// Every coefficient is an integer on one grid 2^emin (at least 55 significant bits relative to
// the largest), every row an exact integer sum rounded once, as in the general kernels. Several
// right-hand sides run as columns of one launch, each with its own scale and copy of x.
// Bound: integer issue and the latency of the table -> element reads. Disordered chains, N = L/2, one
// product in FP64 (before: 128-bit multiply-adds, partners one at a time behind block barriers):
// 24 sites 176 -> 124 us, 26 sites 675 -> 393 us (FP32 172 -> 96, 632 -> 278 us); 5 x 5 lattice with a
// coupling per bond 1090 -> 799 us (FP32 1052 -> 589 us).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <vector>

#include <cuda_runtime.h>

#include "dq_fixed.cuh"
#include "dq_internal.h"

namespace dq {

constexpr int kPBT = 256;  // threads per CTA

int build_panel_pb(const dq_sector* s, double C, const double* lin,
                   const std::vector<std::pair<std::pair<int, int>, std::pair<double, double>>>& pairs, dq_terms* t) {
    t->pb_ok = false;
    if (s->Q != 2 || s->n_sub != 2 || s->wide) return DQ_OK;
    const int L0 = s->Lk[0], L1 = s->Lk[1], N = s->N, L = s->L;
    if (L1 < 1 || L1 > kPBMaxL1 || L0 > 16) return DQ_OK;
    PanelPB& P = t->pbp;
    std::memset(&P, 0, sizeof P);
    P.L0 = L0;
    P.L1 = L1;
    P.N = N;
    struct Bond {
        int lo, hi;
        double A, K;
    };
    std::vector<Bond> all;
    std::vector<std::pair<uint32_t, double>> p0hop;  // (s0 pair mask, amplitude)
    std::vector<double> p1A, xA;
    std::map<uint32_t, std::vector<std::pair<uint32_t, double>>> xh;  // P_0 bit a -> (P_1 bit b, A)
    double cmax = std::fabs(C);
    int nzz = 0, np1 = 0, nxz = 0;
    for (auto& e : pairs) {
        const int lo = e.first.first, hi = lo + e.first.second;
        const double K = e.second.first, A = e.second.second;
        if (K == 0.0 && A == 0.0) continue;
        all.push_back({lo, hi, A, K});
        cmax = std::max(cmax, std::max(std::fabs(K), std::fabs(A)));
        if (K != 0.0) ++nzz;
        if (hi < L1) {
            if (np1++ == kPBMaxBonds) return DQ_OK;
            if (A == 0.0) continue;
            P.p1_lo2[P.n1b] = 2u << lo;
            P.p1_d[P.n1b] = hi - lo;
            P.p1_pm2[P.n1b++] = (2u << lo) | (2u << hi);
            p1A.push_back(A);
        } else if (lo >= L1) {
            if (A != 0.0) p0hop.push_back({(1u << (lo - L1)) | (1u << (hi - L1)), A});
        } else {
            if (A != 0.0) xh[1u << (hi - L1)].push_back({2u << lo, A});
            if (K != 0.0 && nxz++ == kPBMaxBonds) return DQ_OK;
        }
    }
    if ((int)xh.size() > kPBMaxGroups || p0hop.size() > 200) return DQ_OK;
    for (int p = 0; p < L; ++p) cmax = std::max(cmax, std::fabs(lin[p]));
    // one grid 2^emin for all coefficients; a row's diagonal (1 + L + nzz unit terms) stays
    // below 2^62, each hop amplitude below 2^55
    long long tdiag = 1 + L + nzz;
    int lg = 0;
    while ((1ll << lg) < tdiag) ++lg;
    const int mbits = std::min(55, 62 - lg);
    P.emin = cmax > 0.0 ? std::ilogb(cmax) + 1 - mbits : 0;
    auto M = [&](double c) { return (long long)std::llrint(std::ldexp(c, -P.emin)); };
    for (auto& g : xh) {
        P.xg_abit[P.nxg] = g.first;
        P.xg_first[P.nxg] = P.nvis;
        for (auto& e : g.second) {
            if (P.nvis == kPBMaxBonds) return DQ_OK;
            P.xb_bit2[P.nvis++] = e.first;
            xA.push_back(e.second);
        }
        P.xg_end[P.nxg++] = P.nvis;
    }
    // most hops one row can have (a pair differs only between an occupied and an empty site)
    {
        auto most = [](size_t bonds, int sites) { return std::min(bonds, (size_t)(sites / 2) * ((sites + 1) / 2)); };
        P.flush = most(p0hop.size(), L0) + most(p1A.size(), L1) + xA.size() > 63;
    }
    std::vector<int2> amp;
    auto add_amp = [&](double c) {
        const long long m = M(c), hi = (m + (1ll << 27)) >> 28;
        amp.push_back(make_int2((int)hi, (int)(m - hi * (1ll << 28))));
    };
    for (double c : p1A) add_amp(c);
    for (double c : xA) add_amp(c);
    for (auto& e : p0hop) add_amp(e.second);
    P.namp = (int)amp.size();
    // P_1 tables (local index within its particle-number sector, the states per sector)
    const auto& rt = s->h.rank_tab[s->dev.tab[1]];
    const auto& ut = s->h.unrank_tab[s->dev.tab[1]];
    const auto& ss = s->h.sec_start[s->dev.tab[1]];
    std::vector<uint16_t> t1rank(rt.size()), t1states(ut.size());
    for (size_t q = 0; q < rt.size(); ++q) t1rank[q] = (uint16_t)(rt[q] == 0xffffffffu ? 0 : rt[q]);
    for (size_t q = 0; q < ut.size(); ++q) t1states[q] = (uint16_t)ut[q];
    for (int n = 0; n <= L1 + 1; ++n) {
        P.t1start[n] = ss[n <= L1 ? n : L1 + 1];
        P.t1len[n] = n <= L1 ? ss[n + 1] - ss[n] : 0;
    }
    // Sz Sz bonds by place and fields, as integers
    struct Zz {
        uint32_t lo, hi;  // bits (in s1 or s0)
        long long K;
    };
    std::vector<Zz> z1, z0, zx;
    for (const Bond& e : all) {
        if (e.K == 0.0) continue;
        if (e.hi < L1)
            z1.push_back({(uint32_t)e.lo, (uint32_t)e.hi, M(e.K)});
        else if (e.lo >= L1)
            z0.push_back({(uint32_t)(e.lo - L1), (uint32_t)(e.hi - L1), M(e.K)});
        else
            zx.push_back({(uint32_t)e.lo, (uint32_t)(e.hi - L1), M(e.K)});
    }
    std::vector<long long> ml(L);
    for (int b = 0; b < L; ++b) ml[b] = M(lin[b]);
    std::vector<long long> d1(t1states.size(), 0);
    for (size_t q = 0; q < t1states.size(); ++q) {
        const uint32_t w = t1states[q];
        long long d = 0;
        for (const Zz& e : z1) d += (((w >> e.lo) ^ (w >> e.hi)) & 1u) ? e.K : 0;
        for (uint32_t m = w; m; m &= m - 1) d += ml[__builtin_ctz(m)];
        d1[q] = d;
    }
    // panels (longest first, so that the last ones of a launch are short; canonical inside a length),
    // their diagonal and sources
    const auto& u0 = s->h.unrank_tab[s->dev.tab[0]];
    const auto& s0s = s->h.sec_start[s->dev.tab[0]];
    std::vector<uint32_t> ps0;
    std::vector<uint64_t> pst, lst;
    std::vector<PanelRowDiag> pdiag;
    std::vector<uint32_t> loff, lhdr;
    const long long MC = M(C);
    std::vector<std::pair<uint32_t, uint32_t>> pl;  // (~length, s0)
    pl.reserve(u0.size());
    for (int n0 = 0; n0 <= L0; ++n0) {
        const int n1 = N - n0;
        if (n1 < 0 || n1 > L1) continue;
        P.cmax = std::max(P.cmax, (int)P.t1len[n1]);
        for (uint32_t q = s0s[n0]; q < s0s[n0 + 1]; ++q) pl.push_back({~P.t1len[n1], u0[q]});
    }
    std::stable_sort(pl.begin(), pl.end(), [](auto& a, auto& b) { return a.first < b.first; });
    pdiag.reserve(pl.size());
    lst.reserve(pl.size() * (p0hop.size() / 2 + P.nxg + 1));
    for (auto& e : pl) {
        const uint32_t s0 = e.second;
        const uint64_t start = s->h.c0_tab[s0];
        if (start >> 48) return DQ_OK;
        ps0.push_back(s0);
        pst.push_back(start);
        PanelRowDiag g;
        std::memset(&g, 0, sizeof g);
        g.pd = MC;
        for (uint32_t m = s0; m; m &= m - 1) g.pd += ml[L1 + __builtin_ctz(m)];
        for (const Zz& e : z0) g.pd += (((s0 >> e.lo) ^ (s0 >> e.hi)) & 1u) ? e.K : 0;
        for (const Zz& e : zx) {
            const bool sa = (s0 >> e.hi) & 1u;
            g.pd += sa ? e.K : 0;
            g.w[e.lo] += sa ? -e.K : e.K;
        }
        pdiag.push_back(g);
        loff.push_back((uint32_t)lst.size());
        uint32_t n0p = 0, nx = 0;
        for (size_t b = 0; b < p0hop.size(); ++b)
            if (__builtin_popcount(s0 & p0hop[b].first) == 1) {
                lst.push_back(s->h.c0_tab[s0 ^ p0hop[b].first] | ((uint64_t)b << 48));
                ++n0p;
            }
        for (int g2 = 0; g2 < P.nxg; ++g2) {
            const uint64_t src = s->h.c0_tab[s0 ^ P.xg_abit[g2]];
            if (src == UINT64_MAX) continue;  // no partner sector: no row of the panel hops here
            lst.push_back(src | ((uint64_t)g2 << 48));
            ++nx;
        }
        lhdr.push_back(n0p | (nx << 8));
    }
    loff.push_back((uint32_t)lst.size());
    P.npanels = (uint32_t)ps0.size();
    int rc;
    void* p;
#define DQ_UP(vec, field, type)                                                                   \
    if ((rc = dev_upload(t->dev_allocs, vec.data(), vec.size() * sizeof(vec[0]), &p))) return rc; \
    P.field = (const type*)p;
    DQ_UP(ps0, panel_s0, uint32_t)
    DQ_UP(pst, panel_start, uint64_t)
    DQ_UP(t1rank, t1rank, uint16_t)
    DQ_UP(t1states, t1states, uint16_t)
    DQ_UP(amp, amp, int2)
    DQ_UP(d1, d1, long long)
    DQ_UP(pdiag, pdiag, PanelRowDiag)
    DQ_UP(loff, list_off, uint32_t)
    DQ_UP(lhdr, list_hdr, uint32_t)
    DQ_UP(lst, list, uint64_t)
#undef DQ_UP
    t->pb_ok = true;
    return DQ_OK;
}

// ------------------------------------------------------------------ device ------------------

// A row's hop sum. float64 vectors: X split in two 32-bit halves (split_word), four 32 x 32 -> 64-bit
// multiply-adds per hop, each sum below 2^56 per hop; float32 vectors: 31-bit X, two multiply-adds,
// below 2^57 per hop: 63 hops fit (a 64 x 64 -> 128-bit multiply-add per hop took about 25 instructions).
template <typename XT>
struct PBSum;
template <>
struct PBSum<long long> {
    Acc3 a;
    __device__ __forceinline__ void init() { a = {0, 0, 0}; }
    __device__ __forceinline__ void add(int2 m, long long x) { acc_hop(a, m, x); }
    __device__ __forceinline__ void total(I128& r) const {
        add_shifted(r, a.hh, 56);
        add_shifted(r, a.mid, 28);
        add_shifted(r, a.ll, 0);
    }
    __device__ __forceinline__ static long long value(long long x) { return join_word(x); }
};
template <>
struct PBSum<int> {
    long long hi, lo;
    __device__ __forceinline__ void init() { hi = lo = 0; }
    __device__ __forceinline__ void add(int2 m, int x) {
        hi = mad_wide(m.x, x, hi);
        lo = mad_wide(m.y, x, lo);
    }
    __device__ __forceinline__ void total(I128& r) const {
        add_shifted(r, hi, 28);
        add_shifted(r, lo, 0);
    }
    __device__ __forceinline__ static long long value(int x) { return x; }
};

template <typename XT>
__device__ __forceinline__ XT pb_lds(const unsigned char* base, uint32_t off) {
    return *reinterpret_cast<const XT*>(base + off);
}

// Asynchronous copy of one element into shared memory.
template <typename XT>
__device__ __forceinline__ void pb_copy(XT* dst, const XT* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(sizeof(XT))
                 : "memory");
}
__device__ __forceinline__ void pb_copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int kPBSlots = 4;              // cut partner panels held at a time
constexpr int kPBLow = 128, kPBSums = kPBLow + 64;  // diagonal sums by the low seven P_1 bits, by the others
constexpr int kPBList = 256;             // sources of a panel

// Shared memory: the rank table (2^L1 + 8 u16 byte offsets, entry 2^L1 points at a zero element), the
// panel's own x and up to kPBSlots partner panels (cap + 8 elements each), the amplitudes, the diagonal
// sums, the source lists of this panel and of the next one.
template <typename XT>
struct PBSmem {
    int own, bstride, amp, sums, lst, slots, total;
    __host__ __device__ PBSmem(const PanelPB& P, int cap) {
        auto al = [](int b) { return (b + 127) & ~127; };
        slots = P.nxg < kPBSlots ? P.nxg : kPBSlots;
        own = al((1 << P.L1) * 2 + 16);
        bstride = al((cap + 8) * (int)sizeof(XT));
        amp = own + (1 + slots) * bstride;
        sums = al(amp + P.namp * 8);
        lst = sums + kPBSums * 8;
        total = lst + 2 * kPBList * 8;
    }
};

// What a block reads of a panel one panel ahead.
struct PBHead {
    uint64_t start;
    uint32_t s0, hdr, pi;
    int col;
};

template <typename XT, typename OUT, int E, bool FLUSH>
__device__ __forceinline__ void pb_rows(const PanelPB& P, const PBSmem<XT>& L, const XT* __restrict__ X,
                                        OUT* __restrict__ y, int ld, unsigned char* smem, const PBHead& hd, int scale) {
    using Sum = PBSum<XT>;
    constexpr int U = sizeof(XT) == 8 ? 2 : 4;  // P_0 partners in flight
    const int tid = threadIdx.x;
    const uint32_t s0 = hd.s0;
    const int n1 = P.N - __popc(s0), C = (int)P.t1len[n1], np0 = (int)(hd.hdr & 255u), nx = (int)((hd.hdr >> 8) & 255u);
    const uint64_t* lst = reinterpret_cast<const uint64_t*>(smem + L.lst);
    const int2* amp = reinterpret_cast<const int2*>(smem + L.amp);
    unsigned char* own = smem + L.own;
    const uint16_t* states = P.t1states + P.t1start[n1];
    uint32_t s2[E];  // P_1 pattern of each row, shifted left by one (rank-table byte offset)
    Sum acc[E];
    I128 big[FLUSH ? E : 1];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = tid + e * kPBT;
        s2[e] = c < C ? (uint32_t)__ldg(states + c) << 1 : 0u;
        acc[e].init();
        if (FLUSH) big[e] = {0, 0};
    }
    auto flush = [&]() {
        if constexpr (FLUSH) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                acc[e].total(big[e]);
                acc[e].init();
            }
        }
    };
    // hops inside P_0: partner panels element by element, while the copies of the panel's own x and of
    // the cut partners land
    const int2* amp0 = amp + P.n1b + P.nvis;
    for (int l = 0; l < np0; l += U) {
        const XT* src[U];
        int2 m[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t ent = lst[min(l + u, np0 - 1)];
            src[u] = X + (ent & ((1ull << 48) - 1));
            m[u] = l + u < np0 ? amp0[ent >> 48] : make_int2(0, 0);
        }
        XT v[U][E];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int e = 0; e < E; ++e) v[u][e] = tid + e * kPBT < C ? __ldg(src[u] + tid + e * kPBT) : (XT)0;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e].add(m[u], v[u][e]);
        if (FLUSH && l % 56 == 56 - U) flush();
    }
    flush();
    pb_copies_done();
    __syncthreads();
    // hops inside P_1 through the rank table; a pair that is not active reads the zero element
    const uint32_t zslot = 2u << P.L1;
    for (int q = 0; q < P.n1b; ++q) {
        const uint32_t lo2 = P.p1_lo2[q], pm2 = P.p1_pm2[q];
        const int d = P.p1_d[q];
        const int2 m = amp[q];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const uint32_t t = ((s2[e] ^ (s2[e] >> d)) & lo2) ? s2[e] ^ pm2 : zslot;
            acc[e].add(m, pb_lds<XT>(own, pb_lds<uint16_t>(smem, t)));
        }
        if (FLUSH && q % 56 == 55) flush();
    }
    flush();
    // hops across the cut: the partner panels in the slots, kPBSlots at a time
    for (int j0 = 0; j0 < nx; j0 += kPBSlots) {
        if (j0) {
            __syncthreads();  // the slots' previous partners are no longer read
            for (int j = j0; j < min(j0 + kPBSlots, nx); ++j) {
                const uint64_t ent = lst[np0 + j];
                const int len = (int)P.t1len[(s0 & P.xg_abit[ent >> 48]) ? n1 + 1 : n1 - 1];
                XT* dst = reinterpret_cast<XT*>(own + (1 + j - j0) * L.bstride);
                for (int c = tid; c < len; c += kPBT) pb_copy(dst + c, X + (ent & ((1ull << 48) - 1)) + c);
            }
            pb_copies_done();
            __syncthreads();
        }
        for (int j = j0; j < min(j0 + kPBSlots, nx); ++j) {
            const int g = (int)(lst[np0 + j] >> 48);
            const unsigned char* slot = own + (1 + j - j0) * L.bstride;
            const uint32_t flip = (s0 & P.xg_abit[g]) ? ~0u : 0u;  // the hop needs s_b != s_a
            for (int q = P.xg_first[g]; q < P.xg_end[g]; ++q) {
                const uint32_t bb2 = P.xb_bit2[q];
                const int2 m = amp[P.n1b + q];
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const uint32_t t = ((s2[e] ^ flip) & bb2) ? s2[e] ^ bb2 : zslot;
                    acc[e].add(m, pb_lds<XT>(slot, pb_lds<uint16_t>(smem, t)));
                }
            }
            flush();
        }
    }
    // the row result: d x_i + sum of the hops, exactly, rounded once
    const long long* sums = reinterpret_cast<const long long*>(smem + L.sums);
    const long long* d1 = P.d1 + P.t1start[n1];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = tid + e * kPBT;
        if (c >= C) continue;
        const uint32_t s = s2[e] >> 1;
        const long long md = __ldg(d1 + c) + sums[s & (kPBLow - 1)] + sums[kPBLow + (s >> 7)];
        I128 r = {0, 0};
        if (FLUSH) r = big[FLUSH ? e : 0];
        mac(r, md, Sum::value(pb_lds<XT>(own, (uint32_t)(c * sizeof(XT)))));
        acc[e].total(r);
        y[(hd.start + c) * ld + hd.col] = i128_to<OUT>(r, scale);
    }
}

// Three CTAs per SM (at most 80 registers per thread). Items: panel * cols + column, so that the columns
// of a panel, which write the same lines of y, run side by side. xstride: elements of X per column.
template <typename XT, typename OUT, bool FLUSH>
__global__ void __launch_bounds__(kPBT, FLUSH ? 2 : 3)
    k_panel_pb(PanelPB P, PBSmem<XT> L, const XT* __restrict__ X, OUT* __restrict__ y, const ColScale* __restrict__ h,
               int* err, int cap, uint64_t D, uint64_t xstride, int cols) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ PBHead next;
    const int tid = threadIdx.x;
    uint16_t* t1 = reinterpret_cast<uint16_t*>(smem);
    uint64_t* lst = reinterpret_cast<uint64_t*>(smem + L.lst);
    const uint32_t ntab = 1u << P.L1;
    for (uint32_t q = tid; q <= ntab; q += kPBT)
        t1[q] = (uint16_t)((q < ntab ? (uint32_t)__ldg(P.t1rank + q) : (uint32_t)cap) * sizeof(XT));
    for (int q = tid; q < 8 * (1 + L.slots); q += kPBT) reinterpret_cast<XT*>(smem + L.own + (q / 8) * L.bstride)[cap + q % 8] = 0;
    for (int q = tid; q < P.namp; q += kPBT) reinterpret_cast<int2*>(smem + L.amp)[q] = __ldg(P.amp + q);
    if (h->bad) {  // an Inf or NaN in x: y is NaN and the error word is raised
        for (uint64_t i = blockIdx.x * (uint64_t)kPBT + tid; i < D * cols; i += (uint64_t)gridDim.x * kPBT) y[i] = (OUT)NAN;
        if (blockIdx.x == 0 && tid == 0) atomicAdd(err, 1);
        return;
    }
    // the last warp reads the head and the source list of the next item into `next`
    const uint64_t items = (uint64_t)P.npanels * cols;
    auto fetch = [&](uint64_t item) {
        if (tid < kPBT - 32 || item >= items) return;
        const int lane = tid & 31;
        const uint32_t pi = (uint32_t)(item / cols);
        const uint32_t lo = __ldg(P.list_off + pi), hi = __ldg(P.list_off + pi + 1);
        for (uint32_t q = lo + lane; q < hi; q += 32) lst[kPBList + q - lo] = __ldg(P.list + q);
        if (lane == 0) {
            next.s0 = __ldg(P.panel_s0 + pi);
            next.start = __ldg(P.panel_start + pi);
            next.hdr = __ldg(P.list_hdr + pi);
            next.pi = pi;
            next.col = (int)(item % cols);
        }
    };
    fetch(blockIdx.x);
    for (uint64_t item = blockIdx.x; item < items; item += gridDim.x) {
        __syncthreads();  // the previous item is finished, the next one's head and list are there
        const PBHead hd = next;
        const XT* Xc = X + hd.col * xstride;
        const int n1 = P.N - __popc(hd.s0), C = (int)P.t1len[n1];
        const int np0 = (int)(hd.hdr & 255u), nx = (int)((hd.hdr >> 8) & 255u);
        XT* own = reinterpret_cast<XT*>(smem + L.own);
        for (int c = tid; c < C; c += kPBT) pb_copy(own + c, Xc + hd.start + c);
        for (int j = 0; j < min(nx, kPBSlots); ++j) {
            const uint64_t ent = lst[kPBList + np0 + j];
            const int len = (int)P.t1len[(hd.s0 & P.xg_abit[ent >> 48]) ? n1 + 1 : n1 - 1];
            XT* dst = reinterpret_cast<XT*>(smem + L.own + (1 + j) * L.bstride);
            for (int c = tid; c < len; c += kPBT) pb_copy(dst + c, Xc + (ent & ((1ull << 48) - 1)) + c);
        }
        for (int q = tid; q < np0 + nx; q += kPBT) lst[q] = lst[kPBList + q];
        if (tid < kPBSums) {
            const PanelRowDiag* pd = P.pdiag + hd.pi;
            long long sum = tid < kPBLow ? __ldg(&pd->pd) : 0;
            const long long* w = pd->w + (tid < kPBLow ? 0 : 7);
#pragma unroll
            for (int q = 0; q < 7; ++q)
                if ((tid >> q) & (tid < kPBLow ? 1 : q < 6)) sum += __ldg(w + q);
            reinterpret_cast<long long*>(smem + L.sums)[tid] = sum;
        }
        __syncthreads();
        fetch(item + gridDim.x);
        const int scale = P.emin - h->F[hd.col];
#define PB_ROWS(e) pb_rows<XT, OUT, e, FLUSH>(P, L, Xc, y, cols, smem, hd, scale)
        switch ((C + kPBT - 1) / kPBT) {
            case 7: PB_ROWS(7); break;
            case 6: PB_ROWS(6); break;
            case 5: PB_ROWS(5); break;
            case 4: PB_ROWS(4); break;
            case 3: PB_ROWS(3); break;
            case 2: PB_ROWS(2); break;
            default: PB_ROWS(1);
        }
#undef PB_ROWS
    }
}

// Column c of the interleaved x as fixed point at X + c * xstride (float64: split words).
template <typename T, typename XT>
__global__ void k_pb_fixed(const T* __restrict__ x, XT* __restrict__ X, uint64_t n, int cols, uint64_t xstride, ColScale* h) {
    using U = typename FBits<T>::U;
    const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
    const int c = (int)(t0 % (uint64_t)cols);  // step is a multiple of cols: a thread stays on one column
    const int emax = h->emax[c];
    const int F = XHead<XT>::HEAD - (emax - FBits<T>::BIAS + 1);
    if (t0 < (uint64_t)cols) {
        h->F[c] = F;
        if (emax == FBits<T>::EMASK) h->bad = 1;  // Inf or NaN in column c
    }
    if (emax == FBits<T>::EMASK) return;
#pragma unroll 4
    for (uint64_t i = t0; i < n; i += step) {
        const XT v = to_fixed<T, XT>(reinterpret_cast<const U*>(x)[i], F);
        const uint64_t at = cols == 1 ? i : c * xstride + i / cols;
        if constexpr (sizeof(XT) == 8)
            X[at] = split_word(v);
        else
            X[at] = v;
    }
}

template <typename T, typename XT, bool FLUSH>
static int run_pb(const dq_sector* s, dq_terms* t, const T* x, T* y, int cols, cudaStream_t st) {
    const PanelPB& P = t->pbp;
    const uint64_t xstride = (s->D + 15) & ~15ull;
    const size_t need = kColScaleBytes + (size_t)xstride * cols * sizeof(XT);
    if (t->scratch_bytes < need) {
        if (t->scratch) cudaFree(t->scratch);
        t->scratch = nullptr;
        t->scratch_bytes = 0;
        cudaError_t e = cudaMalloc(&t->scratch, need);
        if (e != cudaSuccess) return (int)e;
        t->scratch_bytes = need;
    }
    ColScale* h = reinterpret_cast<ColScale*>(t->scratch);
    XT* X = reinterpret_cast<XT*>(reinterpret_cast<char*>(t->scratch) + kColScaleBytes);
    cudaMemsetAsync(h, 0, sizeof(ColScale), st);
    const int sms = sm_count_cached(), bs = col_block(cols);
    const uint64_t n = s->D * (uint64_t)cols;
    const unsigned pgrid = (unsigned)std::min<uint64_t>((n + bs - 1) / bs, (uint64_t)sms * 8);
    if (cols == 1)
        k_exp_max<T><<<pgrid, 256, 0, st>>>(x, n, reinterpret_cast<WsHeader*>(h));  // emax[0] is its first word
    else
        k_col_exp_max<T><<<pgrid, bs, 0, st>>>(x, n, cols, h);
    k_pb_fixed<T, XT><<<pgrid, bs, 0, st>>>(x, X, n, cols, xstride, h);
    const int cap = P.cmax;
    const PBSmem<XT> L(P, cap);
    auto kern = k_panel_pb<XT, T, FLUSH>;
    if (L.total > 40 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L.total);
        if (e != cudaSuccess) return (int)e;
    }
    const int per_sm = occupancy_cached(reinterpret_cast<const void*>(kern), kPBT, L.total);
    const uint64_t items = (uint64_t)P.npanels * cols;
    const unsigned grid = (unsigned)std::min<uint64_t>(std::max<uint64_t>(items, 1), (uint64_t)sms * per_sm);
    const int tslot = timing_start(st);
    kern<<<grid, kPBT, L.total, st>>>(P, L, X, y, h, s->dev.err, cap, s->D, xstride, cols);
    timing_stop(tslot, st, 3);
    return (int)cudaGetLastError();
}

int launch_panel_pb(const dq_sector* s, dq_terms* t, const void* x, void* y, int dtype, int cols, void* stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const bool fl = t->pbp.flush;
    if (dtype == DQ_F64)
        return fl ? run_pb<double, long long, true>(s, t, (const double*)x, (double*)y, cols, st)
                  : run_pb<double, long long, false>(s, t, (const double*)x, (double*)y, cols, st);
    return fl ? run_pb<float, int, true>(s, t, (const float*)x, (float*)y, cols, st)
              : run_pb<float, int, false>(s, t, (const float*)x, (float*)y, cols, st);
}

}  // namespace dq

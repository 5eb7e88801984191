// Host side of the panel product: decides whether it applies and builds its plan.
//
// With two subsystems the canonical index is c_0(s0) + index_1(s1) (Sec. 3.3, Lin's two tables),
// so all states with one P_0 pattern s0 occupy a contiguous range of D_2(L_1, N - n_0) indices,
// ordered by the local index of s1. A bond between sites i < j acts on such "panels" in one of
// three ways:
//   both sites in P_1:  a permutation inside the panel, the same for every panel of a block;
//   both sites in P_0:  panel s0 receives panel s0' (two bits swapped) element by element;
//   across the cut:     panel s0 receives panel s0 ^ bit_a (the neighbouring particle-number
//                       block) through the map s1 -> index_1(s1 ^ bit_b).
// Requirements: Q = 2, two subsystems, L_1 <= 15 (panels of at most 6435 rows), uniform
// single-site fields, at most two distinct hop amplitudes and four distinct coefficients of
// [s_i != s_j], and coefficients that are small integer multiples of one power of two.
//
// With three or more subsystems the same holds with P_0 = all subsystems but the last and P_1 =
// the last one (Eq. (index): the last subsystem has offset 0 and stride 1 inside the block of its
// particle number, so the rows sharing the prefix pattern s0 are again contiguous, in P_1's local
// order). Those panels are small (P_1 of 8 to 10 sites: at most 252 rows) and many, so the
// warp-panel kernel (dq_panel_w.cu) gives each panel one warp and ranks the partner panels on the
// device; the host builds only the panel list and the bond tables. Two subsystems whose P_1 has 8
// to 10 sites take that kernel too.
//
// Three or more subsystems whose last one is shorter than 8 (or longer than 10) sites use P_1 =
// the last TWO subsystems (the "tail") in the panel kernel instead: with the prefix pattern s0
// fixed, the canonical key (n_0, σ0, ..., n_{n-2}, σ_{n-2}, n_{n-1}, σ_{n-1}) leaves only the
// tail's two entries free, so those rows are again one contiguous range, ordered by the tail's
// own two-subsystem canonical order (Eq. (index) restricted to the tail). That order depends on
// the tail's particle number only; the host tabulates it (tail pattern -> local index) from the
// sector's own rank and checks every panel's first and last row.
//
// Large sectors whose own panels are of fewer than 15 sites take neither (use_split_order below has the
// rule): the panel kernel works on x in
// the order of a split into TWO subsystems of its own (the "split order": P_0 = the upper L - L_1 sites,
// P_1 the lower L_1 <= 15), whatever the sector's partition is. The prepass that makes the fixed-point
// copy of x gathers it into that order and the kernel's stores go back through the same map. A panel of
// the split order is a few contiguous pieces of the canonical order: the suffix bits that lie in whole
// subsystems (Llow of them) run through a contiguous range whose order depends on their particle
// number only, one piece per pattern of the suffix bits above. One short panel per warp (k_panel_w),
// or a tail of two short subsystems, reads about 50 partner panels per panel where 15 sites read 34.
// 6 x 5 lattice, N = 15: three subsystems, FP32 21.3 -> 9.5 ms a product; five, FP64 23.4 -> 13.2 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <set>
#include <vector>

#include "dq_internal.h"

namespace dq {

constexpr uint64_t kSplitMinDim = 1ull << 19;

// Exponent of the lowest set bit of v's mantissa: v = m * 2^e with m odd.
static int low_exponent(double v) {
    int ex;
    double f = std::frexp(std::fabs(v), &ex);  // |v| = f 2^ex, f in [0.5, 1)
    long long m = (long long)std::ldexp(f, 53);
    int e = ex - 53;
    while ((m & 1) == 0) {
        m >>= 1;
        ++e;
    }
    return e;
}

// The rest of the plan for three or more subsystems: the panel list (every prefix pattern s0
// whose P_1 particle number N - |s0| fits, with its first index), the prefix masks
// of the cut Sz Sz bonds per class and position b, the sector view for the device rank.
static int build_panel_w(const dq_sector* s, PanelPlan& P, const std::vector<uint16_t>& t1rank,
                         const std::vector<uint16_t>& t1states,
                         const std::vector<std::pair<int, std::pair<uint32_t, uint32_t>>>& xz, dq_terms* t) {
    const int L1 = P.L1, L0 = P.L0, N = P.N, last = s->n_sub - 1;
    const int tl = s->dev.tab[last];
    // panels grouped by length (the warps in flight then run one row-count variant of the
    // kernel, which keeps its code in the instruction cache), in canonical order inside a group
    std::vector<std::pair<std::pair<uint32_t, uint64_t>, uint32_t>> pl;  // ((length, start), s0)
    int cmax = 0;
    uint64_t smax = 0;
    for (uint64_t s0 = 0; s0 < (1ull << L0); ++s0) {
        const int n1 = N - __builtin_popcountll(s0);
        if (n1 < 0 || n1 > L1) continue;
        const uint32_t first = s->h.unrank_tab[tl][s->h.sec_start[tl][n1]];  // local index 0
        const u128 w = ((u128)s0 << L1) | first;
        const uint64_t st = host_rank(s, w);
        pl.push_back({{P.t1len[n1], st}, (uint32_t)s0});
        cmax = std::max(cmax, (int)P.t1len[n1]);
        smax = std::max(smax, st);
    }
    std::sort(pl.begin(), pl.end());
    if (pl.empty() || smax >> 48) return DQ_OK;
    std::vector<uint32_t> ps0(pl.size());
    std::vector<uint64_t> pst(pl.size());
    for (size_t q = 0; q < pl.size(); ++q) {
        pst[q] = pl[q].first.second;
        ps0[q] = pl[q].second;
    }
    P.npanels = (uint32_t)pl.size();
    P.cmax = cmax;
    std::memset(P.xzA, 0, sizeof P.xzA);
    for (auto& e : xz) P.xzA[e.first][__builtin_ctz(e.second.second)] |= e.second.first;
    PWRank& R = t->pwr;
    std::memset(&R, 0, sizeof R);
    R.n_sub = s->n_sub;
    R.N = N;
    R.L1 = L1;
    R.os_total = s->dev.os_total;
    R.D = s->D;
    for (int k = 0; k < s->n_sub; ++k) {
        R.shift[k] = s->dev.shift[k];
        R.os_base[k] = s->dev.os_base[k];
        R.os_ld[k] = s->dev.os_ld[k];
        R.fmask[k] = (uint32_t)((1ull << s->Lk[k]) - 1);
        R.rank[k] = s->dev.rank_tab[s->dev.tab[k]];
    }
    R.off = s->dev.off;
    R.str = s->dev.str;
    int rc;
    void* p;
    if ((rc = dev_upload(t->dev_allocs, ps0.data(), ps0.size() * 4, &p))) return rc;
    P.panel_s0 = (const uint32_t*)p;
    if ((rc = dev_upload(t->dev_allocs, pst.data(), pst.size() * 8, &p))) return rc;
    P.panel_start = (const uint64_t*)p;
    if ((rc = dev_upload(t->dev_allocs, t1rank.data(), t1rank.size() * 2, &p))) return rc;
    P.t1rank = (const uint16_t*)p;
    if ((rc = dev_upload(t->dev_allocs, t1states.data(), t1states.size() * 2, &p))) return rc;
    P.t1states = (const uint16_t*)p;
    t->pw_ok = true;
    return DQ_OK;
}

// P_1 of the split order: as many of the lowest sites as the rank table holds (15), while at least 512
// panels are left.
static int split_sites(const dq_sector* s) { return std::min(15, s->L - 9); }

// The split order pays for its gather of x and its scattered stores where its panels are longer than
// those of the sector's own form (own_sites: P_1 of that form, 0 if it does not fit the operator), and
// from 2^19 rows on. Each product of a panel is an own load of the partner or the rank table with little
// else to do, so the cost of a row falls with the length of the panel: own form against split order, FP64
// and FP32, 5 x 5 lattice (N = 12, P_1 of 12 against 15 sites) 580 -> 369, 576 -> 299 us; 9 x 3 lattice
// (13) 2626 -> 1447, 2379 -> 1169; 7 x 4 lattice (14) 3519 -> 2946, 3048 -> 2354; chain of 24 sites (12)
// 103 -> 90, 99 -> 80; chain of 22 sites, 0.7 M rows (11 against 13) 54 -> 47, 49 -> 43. Of equal length
// the own form is faster (7 x 4 with P_1 of 14 sites in the split order: 3569 and 3104).
//
// A block's frame around a panel is the same for a short one, so where the alternative is not this kernel
// with fewer sites (own_panel) but one warp per panel or the general kernel, the panels have to hold 320
// rows on average. J1-J2 chains with three subsystems, FP64, warp panels against split order: 49 rows (31
// sites, N = 6) 294 / 784 us, 204 rows (28, 7) 313 / 378, 257 (30, 8) 1057 / 1442, 269 (27, 7) 228 / 244,
// 362 (26, 7) 210 / 161, 438 (28, 8) 611 / 499, 1068 (25, 8) 228 / 134; the 9 x 3 lattice (27, 7), general
// kernel against split order, 348 / 471.
constexpr uint64_t kSplitMinRows = 320;
static bool use_split_order(const dq_sector* s, int own_sites, bool own_panel) {
    const int L1 = split_sites(s);
    if (s->D < kSplitMinDim || s->D >= (1ull << 48) || L1 <= 10 || L1 <= own_sites || s->L - L1 > 16) return false;
    if (own_panel) return true;
    uint64_t panels = 0, c = 1;  // c = C(L - L1, n0)
    for (int n0 = 0; n0 <= s->L - L1; ++n0) {
        if (s->N - n0 >= 0 && s->N - n0 <= L1) panels += c;
        c = c * (s->L - L1 - n0) / (n0 + 1);
    }
    return s->D >= kSplitMinRows * panels;
}

// Bits of the lowest whole subsystems inside a suffix of L1 bits (L1 itself when the suffix lies
// inside the last subsystem, whose order is lexicographic).
static int whole_bits(const dq_sector* s, int L1) {
    if (L1 <= s->Lk[s->n_sub - 1]) return L1;
    int low = 0;
    for (int k = s->n_sub - 1; k >= 0 && low + s->Lk[k] <= L1; --k) low += s->Lk[k];
    return low;
}

// Most hops of one amplitude class that a row can have, as a bound: of the bonds between two groups of
// sites those between an occupied and an empty one hop.
static int most_hops(const PanelPlan& P, const std::vector<std::pair<int, uint32_t>>& p0,
                     const std::map<int, std::vector<std::pair<int, int>>>& p1,
                     const std::map<uint32_t, std::vector<std::pair<int, uint32_t>>>& cut) {
    int most = 0;
    for (int k = 0; k < kPanelMaxA; ++k) {
        int b0 = 0, b1 = 0, bx = 0;
        for (auto& e : p0) b0 += e.first == k;
        for (auto& g : p1)
            for (auto& e : g.second) b1 += e.first == k;
        for (auto& g : cut)
            for (auto& e : g.second) bx += e.first == k;
        for (int n0 = std::max(0, P.N - P.L1); n0 <= std::min(P.L0, P.N); ++n0) {
            const int n1 = P.N - n0, e0 = P.L0 - n0, e1 = P.L1 - n1;
            most = std::max(most, std::min(b0, n0 * e0) + std::min(b1, n1 * e1) + std::min(bx, n0 * e1 + n1 * e0));
        }
    }
    return most;
}

// One form of the plan: the sector's own order or the split order. *fits: the operator's bonds and
// coefficients fit the form; with check_only nothing else is done.
static int build_form(const dq_sector* s, double C,
                      const std::vector<std::pair<std::pair<int, int>, std::pair<double, double>>>& pairs, dq_terms* t,
                      bool split, bool check_only, bool* fits) {
    *fits = false;
    // the warp-panel kernel for three or more subsystems, and for two when the panels are small
    // (P_1 of 8 to 10 sites: at most 252 rows, which leave most of a 1024-thread CTA idle)
    const int ns = s->n_sub;
    const bool warp = s->Lk[ns - 1] >= 8 && s->Lk[ns - 1] <= 10;
    const bool tail = ns >= 3 && !warp;  // P_1 = the last two subsystems
    int L1 = tail ? s->Lk[ns - 2] + s->Lk[ns - 1] : s->Lk[ns - 1], L0 = s->L - L1;
    const int N = s->N;
    if (warp) {
        if (ns > kPWMaxSub || L0 > 24) return DQ_OK;
    } else if (L1 > 15 || L1 < 1 || L0 > (tail ? 22 : 16)) {
        return DQ_OK;
    }
    if (split) {
        L1 = split_sites(s);
        L0 = s->L - L1;
    }
    PanelPlan& P = t->pp;
    std::memset(&P, 0, sizeof P);
    P.L0 = L0;
    P.L1 = L1;
    P.N = N;
    std::vector<double> Avals, Kvals;
    auto cls_of = [](std::vector<double>& vals, double v, int maxn) -> int {
        for (size_t q = 0; q < vals.size(); ++q)
            if (vals[q] == v) return (int)q;
        if ((int)vals.size() >= maxn) return -1;
        vals.push_back(v);
        return (int)vals.size() - 1;
    };
    // collect bonds by category, keyed so that iteration order is by class
    std::map<std::pair<int, int>, uint32_t> p1z;                      // (class, d) -> low-position mask
    std::map<int, std::vector<std::pair<int, int>>> p1o;               // d -> (class, lo)
    std::vector<std::pair<int, uint32_t>> p0o, p0z;                   // (class, s0 mask)
    std::map<uint32_t, std::vector<std::pair<int, uint32_t>>> xo;     // a bit -> (class, b bit)
    std::vector<std::pair<int, std::pair<uint32_t, uint32_t>>> xz;    // (class, (a bit, b bit))
    for (auto& e : pairs) {
        int lo = e.first.first, d = e.first.second, hi = lo + d;
        double K = e.second.first, A = e.second.second;
        int ka = -1, kk = -1;
        if (A != 0.0 && (ka = cls_of(Avals, A, kPanelMaxA)) < 0) return DQ_OK;
        if (K != 0.0 && (kk = cls_of(Kvals, K, kPanelMaxK)) < 0) return DQ_OK;
        if (hi < L1) {  // both in P_1
            if (A != 0.0) p1o[d].push_back({ka, lo});
            if (K != 0.0) p1z[{kk, d}] |= 1u << lo;
        } else if (lo >= L1) {  // both in P_0
            uint32_t m = (1u << (lo - L1)) | (1u << (hi - L1));
            if (A != 0.0) p0o.push_back({ka, m});
            if (K != 0.0) p0z.push_back({kk, m});
        } else {  // across the cut: a = hi (in P_0), b = lo (in P_1)
            uint32_t abit = 1u << (hi - L1), bbit = 1u << lo;
            if (A != 0.0) xo[abit].push_back({ka, bbit});
            if (K != 0.0) xz.push_back({kk, {abit, bbit}});
        }
    }
    size_t n_p1b = 0;
    for (auto& e : p1o) n_p1b += e.second.size();
    if ((int)p1o.size() > kPanelMaxLayers || n_p1b > (size_t)kPanelMaxBonds || (int)p1z.size() > kPanelMaxLayers || (int)xo.size() > kPanelMaxGroups ||
        (int)p0o.size() > kPanelMaxBonds || (int)p0z.size() > kPanelMaxBonds || (int)xz.size() > kPanelMaxBonds)
        return DQ_OK;
    std::sort(p0o.begin(), p0o.end());
    std::sort(p0z.begin(), p0z.end());
    std::sort(xz.begin(), xz.end());
    {
        int q = 0;
        for (int k = 0; k < kPanelMaxA; ++k) {
            for (auto& e : p0o)
                if (e.first == k) P.p0_mask[q++] = e.second;
            P.p0_end[k] = q;
        }
        q = 0;
        for (auto& layer : p1o) {
            auto v = layer.second;
            std::sort(v.begin(), v.end());
            const int d = layer.first;
            P.p1l_d[P.n_p1l] = d;
            P.p1l_first[P.n_p1l] = q;
            for (auto& e : v)
                if (e.first == 0) {
                    P.p1b_lobit[q] = 1u << e.second;
                    P.p1b_pm2[q++] = ((1u << e.second) | (1u << (e.second + d))) << 1;
                }
            P.p1l_cut[P.n_p1l] = q;
            for (auto& e : v)
                if (e.first == 1) {
                    P.p1b_lobit[q] = 1u << e.second;
                    P.p1b_pm2[q++] = ((1u << e.second) | (1u << (e.second + d))) << 1;
                }
            P.p1l_end[P.n_p1l++] = q;
        }
        q = 0;
        for (int k = 0; k < kPanelMaxK; ++k) {
            for (auto& e : p0z)
                if (e.first == k) P.p0z_mask[q++] = e.second;
            P.p0z_end[k] = q;
        }
        q = 0;
        for (int k = 0; k < kPanelMaxK; ++k) {
            for (auto& e : p1z)
                if (e.first.first == k) {
                    P.p1z_d[q] = e.first.second;
                    P.p1z_mask[q++] = e.second;
                }
            P.p1z_end[k] = q;
        }
        q = 0;
        for (int k = 0; k < kPanelMaxK; ++k) {
            // at most 7 bonds of one class per (b, value of s_a): the kernel counts them in 3 bit planes
            std::map<uint32_t, int> mult;
            for (auto& e : xz)
                if (e.first == k) {
                    if (++mult[e.second.second] > 7) return DQ_OK;
                    P.xz_abit[q] = e.second.first;
                    P.xz_bbit[q++] = e.second.second;
                }
            P.xz_end[k] = q;
        }
        int nb = 0;
        size_t total = 0;
        for (auto& g : xo) total += g.second.size();
        if (total > (size_t)kPanelMaxBonds) return DQ_OK;
        for (auto& g : xo) {
            auto v = g.second;
            std::sort(v.begin(), v.end());
            P.xg_abit[P.n_xg] = g.first;
            P.xg_first[P.n_xg] = nb;
            for (auto& e : v) {
                if (e.first == 0) P.xb_bit[nb++] = e.second;
            }
            P.xg_cut[P.n_xg] = nb;
            for (auto& e : v) {
                if (e.first == 1) P.xb_bit[nb++] = e.second;
            }
            P.xg_end[P.n_xg++] = nb;
        }
    }
    P.nA = (int)Avals.size();
    P.nK = (int)Kvals.size();
    // common power of two of all coefficients
    std::vector<double> all = Avals;
    all.insert(all.end(), Kvals.begin(), Kvals.end());
    all.push_back(C);
    int emin = 1 << 20;
    for (double v : all)
        if (v != 0.0) emin = std::min(emin, low_exponent(v));
    if (emin == (1 << 20)) emin = 0;
    auto scaled = [&](double v, long long& out) -> bool {
        double m = std::ldexp(v, -emin);
        if (std::fabs(m) >= 9.0e15) return false;  // keep |M| < 2^53 so the sums below stay exact
        out = (long long)m;
        return (double)out == m;
    };
    if (!scaled(C, P.MC)) return DQ_OK;
    for (int k = 0; k < P.nK; ++k)
        if (!scaled(Kvals[k], P.MK[k])) return DQ_OK;
    for (int k = 0; k < P.nA; ++k)
        if (!scaled(Avals[k], P.MA[k])) return DQ_OK;
    P.emin = emin;
    P.fold = most_hops(P, p0o, p1o, xo) > kPanelMaxHops;
    *fits = true;
    if (check_only) return DQ_OK;
    // P_1 tables (local index within its particle-number sector, and the states per sector)
    std::vector<uint16_t> t1rank, t1states;
    if (split) {  // lexicographic inside each particle number
        t1rank.assign((size_t)1 << L1, 0);
        for (int n = 0; n <= L1 + 1 && n < 18; ++n) {
            P.t1start[n] = (uint32_t)t1states.size();
            for (uint32_t w = 0; n <= L1 && w < (1u << L1); ++w)
                if (__builtin_popcount(w) == n) {
                    t1rank[w] = (uint16_t)(t1states.size() - P.t1start[n]);
                    t1states.push_back((uint16_t)w);
                }
            P.t1len[n] = (uint32_t)t1states.size() - P.t1start[n];
        }
    } else if (!tail) {
        const int tl = s->dev.tab[ns - 1];
        const auto& rt = s->h.rank_tab[tl];
        const auto& ut = s->h.unrank_tab[tl];
        const auto& ss = s->h.sec_start[tl];
        t1rank.resize(rt.size());
        t1states.resize(ut.size());
        for (size_t q = 0; q < rt.size(); ++q) t1rank[q] = (uint16_t)(rt[q] == 0xffffffffu ? 0 : rt[q]);
        for (size_t q = 0; q < ut.size(); ++q) t1states[q] = (uint16_t)ut[q];
        for (int n = 0; n <= L1 + 1 && n < 18; ++n) {
            P.t1start[n] = ss[n <= L1 ? n : L1 + 1];
            P.t1len[n] = n <= L1 ? ss[n + 1] - ss[n] : 0;
        }
    } else {
        // the tail's order per particle number n: rank the tail patterns behind one prefix s0
        // with |s0| = N - n and subtract the smallest index
        t1rank.assign((size_t)1 << L1, 0);
        t1states.assign((size_t)1 << L1, 0);
        std::vector<std::vector<uint32_t>> byn(L1 + 1);
        for (uint32_t w = 0; w < (1u << L1); ++w) byn[__builtin_popcount(w)].push_back(w);
        uint32_t at = 0;
        for (int n = 0; n <= L1 + 1 && n < 18; ++n) {
            P.t1start[n] = at;
            P.t1len[n] = 0;
            if (n > L1) continue;
            const int n0 = N - n;
            if (n0 >= 0 && n0 <= L0) {
                const u128 rep = (u128)((1ull << n0) - 1) << L1;
                std::vector<uint64_t> r(byn[n].size());
                uint64_t lo = UINT64_MAX;
                for (size_t q = 0; q < byn[n].size(); ++q) lo = std::min(lo, r[q] = host_rank(s, rep | byn[n][q]));
                std::vector<char> hit(byn[n].size(), 0);
                for (size_t q = 0; q < byn[n].size(); ++q) {
                    const uint64_t c = r[q] - lo;
                    if (c >= byn[n].size() || hit[c]) return DQ_OK;  // not a contiguous range
                    hit[c] = 1;
                    t1rank[byn[n][q]] = (uint16_t)c;
                    t1states[at + c] = (uint16_t)byn[n][q];
                }
            } else {
                for (size_t q = 0; q < byn[n].size(); ++q) {
                    t1rank[byn[n][q]] = (uint16_t)q;
                    t1states[at + q] = (uint16_t)byn[n][q];
                }
            }
            P.t1len[n] = (uint32_t)byn[n].size();
            at += P.t1len[n];
        }
    }
    if (warp && !split) return build_panel_w(s, P, t1rank, t1states, xz, t);
    // panels in canonical order: particle number of P_0, then its local order
    std::vector<uint32_t> ps0;
    std::vector<uint64_t> pst;
    int cmax = 0;
    std::vector<uint64_t> tail_start;  // first index of every prefix pattern's panel (tail form, split order)
    if (split) {
        tail_start.assign((size_t)1 << L0, UINT64_MAX);
        uint64_t at = 0;
        for (int n0 = 0; n0 <= L0; ++n0) {
            const int n1 = N - n0;
            if (n1 < 0 || n1 > L1) continue;
            for (uint32_t s0 = 0; s0 < (1u << L0); ++s0) {
                if (__builtin_popcount(s0) != n0) continue;
                tail_start[s0] = at;
                ps0.push_back(s0);
                pst.push_back(at);
                at += P.t1len[n1];
            }
            cmax = std::max(cmax, (int)P.t1len[n1]);
        }
    } else if (!tail) {
        const auto& u0 = s->h.unrank_tab[s->dev.tab[0]];
        const auto& s0s = s->h.sec_start[s->dev.tab[0]];
        for (int n0 = 0; n0 <= L0; ++n0) {
            int n1 = N - n0;
            if (n1 < 0 || n1 > L1) continue;
            for (uint32_t q = s0s[n0]; q < s0s[n0 + 1]; ++q) {
                uint32_t p = u0[q];
                ps0.push_back(p);
                pst.push_back(s->h.c0_tab[p]);
            }
            cmax = std::max(cmax, (int)P.t1len[n1]);
        }
    } else {
        tail_start.assign((size_t)1 << L0, UINT64_MAX);
        std::vector<std::pair<uint64_t, uint32_t>> pl;
        for (uint32_t s0 = 0; s0 < (1u << L0); ++s0) {
            const int n1 = N - __builtin_popcount(s0);
            if (n1 < 0 || n1 > L1) continue;
            const u128 w = (u128)s0 << L1;
            const uint32_t C1 = P.t1len[n1];
            const uint64_t st = host_rank(s, w | t1states[P.t1start[n1]]);
            // the panel is the contiguous range [st, st + C1) in the tail's order
            if (host_rank(s, w | t1states[P.t1start[n1] + C1 - 1]) != st + C1 - 1) return DQ_OK;
            tail_start[s0] = st;
            pl.push_back({st, s0});
            cmax = std::max(cmax, (int)C1);
        }
        std::sort(pl.begin(), pl.end());
        for (auto& e : pl) {
            ps0.push_back(e.second);
            pst.push_back(e.first);
        }
    }
    auto start_of = [&](uint32_t p) -> uint64_t { return tail_start.empty() ? s->h.c0_tab[p] : tail_start[p]; };
    P.npanels = (uint32_t)ps0.size();
    P.cmax = cmax;
    // per-panel diagonal (see PanelRowDiag) and the P_1 Sz Sz sums of the patterns. A panel's sums are built up
    // over the set bits of s0, lowest first: setting bit a changes [s_a != s_j] of its bonds inside P_0 by
    // 1 - 2 s_j, and turns its bonds across the cut from s_b to 1 - s_b.
    std::vector<PanelRowDiag> pdiag(ps0.size());
    uint32_t nb[32][kPanelMaxK] = {};  // P_0 bits with a bond of class k to bit a
    std::vector<std::vector<std::pair<int, long long>>> cut(32);
    PanelRowDiag none;  // s0 = 0
    std::memset(&none, 0, sizeof none);
    none.pd = P.MC;
    for (int k = 0; k < P.nK; ++k) {
        for (int l = (k ? P.p0z_end[k - 1] : 0); l < P.p0z_end[k]; ++l) {
            const uint32_t lo = P.p0z_mask[l] & (~P.p0z_mask[l] + 1u), hi = P.p0z_mask[l] ^ lo;
            nb[__builtin_ctz(lo)][k] |= hi;
            nb[__builtin_ctz(hi)][k] |= lo;
        }
        for (int l = (k ? P.xz_end[k - 1] : 0); l < P.xz_end[k]; ++l) {
            const int bit = __builtin_ctz(P.xz_bbit[l]);
            none.w[bit] += P.MK[k];
            cut[__builtin_ctz(P.xz_abit[l])].push_back({bit, P.MK[k]});
        }
    }
    for (size_t q = 0; q < ps0.size(); ++q) {
        PanelRowDiag& g = pdiag[q];
        g = none;
        uint32_t below = 0;
        for (uint32_t m = ps0[q]; m; m &= m - 1) {
            const int at = __builtin_ctz(m);
            for (int k = 0; k < P.nK; ++k)
                g.pd += P.MK[k] * (__builtin_popcount(nb[at][k]) - 2 * __builtin_popcount(nb[at][k] & below));
            for (auto& e : cut[at]) {
                g.pd += e.second;
                g.w[e.first] -= 2 * e.second;
            }
            below |= 1u << at;
        }
    }
    std::vector<long long> d1(t1states.size(), 0);
    for (size_t q = 0; q < t1states.size(); ++q)
        for (int k = 0; k < P.nK; ++k)
            for (int l = (k ? P.p1z_end[k - 1] : 0); l < P.p1z_end[k]; ++l)
                d1[q] += P.MK[k] * __builtin_popcount((t1states[q] ^ (t1states[q] >> P.p1z_d[l])) & P.p1z_mask[l]);
    // per-panel source lists
    std::vector<uint32_t> loff(ps0.size() + 1, 0), lhdr(ps0.size(), 0);
    std::vector<uint64_t> lst;
    lst.reserve(ps0.size() * 24);
    for (size_t q = 0; q < ps0.size(); ++q) {
        const uint32_t s0 = ps0[q];
        loff[q] = (uint32_t)lst.size();
        uint32_t cnt[kPanelMaxA] = {0, 0};
        for (int k = 0; k < kPanelMaxA; ++k)
            for (int l = (k ? P.p0_end[k - 1] : 0); l < P.p0_end[k]; ++l) {
                uint32_t m = P.p0_mask[l];
                if (__builtin_popcount(s0 & m) != 1) continue;
                lst.push_back(start_of(s0 ^ m));
                ++cnt[k];
            }
        uint32_t nx = 0;
        for (int g = 0; g < P.n_xg; ++g) {
            uint64_t src = start_of(s0 ^ P.xg_abit[g]);
            if (src == UINT64_MAX) continue;
            if (src >> 48) return DQ_OK;  // indices this large are left to the general kernel
            lst.push_back(src | ((uint64_t)g << 48));
            ++nx;
        }
        lhdr[q] = cnt[0] | (cnt[1] << 8) | (nx << 16);
    }
    loff[ps0.size()] = (uint32_t)lst.size();
    int rc;
    void* p;
    if ((rc = dev_upload(t->dev_allocs, ps0.data(), ps0.size() * 4, &p))) return rc;
    P.panel_s0 = (const uint32_t*)p;
    if ((rc = dev_upload(t->dev_allocs, pst.data(), pst.size() * 8, &p))) return rc;
    P.panel_start = (const uint64_t*)p;
    if ((rc = dev_upload(t->dev_allocs, t1rank.data(), t1rank.size() * 2, &p))) return rc;
    P.t1rank = (const uint16_t*)p;
    if ((rc = dev_upload(t->dev_allocs, t1states.data(), t1states.size() * 2, &p))) return rc;
    P.t1states = (const uint16_t*)p;
    if ((rc = dev_upload(t->dev_allocs, loff.data(), loff.size() * 4, &p))) return rc;
    P.list_off = (const uint32_t*)p;
    if ((rc = dev_upload(t->dev_allocs, lhdr.data(), lhdr.size() * 4, &p))) return rc;
    P.list_hdr = (const uint32_t*)p;
    if ((rc = dev_upload(t->dev_allocs, lst.data(), lst.size() * 8, &p))) return rc;
    P.list = (const uint64_t*)p;
    if ((rc = dev_upload(t->dev_allocs, pdiag.data(), pdiag.size() * sizeof(PanelRowDiag), &p))) return rc;
    P.diag = (const PanelRowDiag*)p;
    if ((rc = dev_upload(t->dev_allocs, d1.data(), d1.size() * 8, &p))) return rc;
    P.d1 = (const long long*)p;
    P.c0 = s->dev.c0_tab;
    if (split) {
        // canonical order of the rows of a panel (see the file comment)
        const int low = whole_bits(s, L1), L = s->L;
        const uint32_t lowmask = (1u << low) - 1;
        P.Llow = low;
        P.npiece = 1 << (L1 - low);
        std::vector<std::vector<uint32_t>> byn(low + 1);
        for (uint32_t w = 0; w <= lowmask; ++w) byn[__builtin_popcount(w)].push_back(w);
        std::vector<uint32_t> pos((size_t)lowmask + 1, 0), rowy(t1states.size());
        for (int n = 0; n <= low; ++n) {
            P.lowfirst[n] = byn[n][0];
            const int up = N - n;
            if (up < 0 || up > L - low) continue;  // no state of the sector has n particles there
            const u128 rep = (((u128)1 << up) - 1) << low;
            std::vector<std::pair<uint64_t, uint32_t>> r;
            for (uint32_t w : byn[n]) r.push_back({host_rank(s, rep | w), w});
            std::sort(r.begin(), r.end());
            for (size_t q = 0; q < r.size(); ++q) {
                if (r[q].first != r[0].first + q) return set_error(DQ_ERANGE, "split order: the suffix is not contiguous");
                pos[r[q].second] = (uint32_t)q;
            }
            P.lowfirst[n] = r[0].second;
        }
        for (size_t q = 0; q < t1states.size(); ++q)
            rowy[q] = pos[t1states[q] & lowmask] | ((uint32_t)(t1states[q] >> low) << 16);
        if ((rc = dev_upload(t->dev_allocs, rowy.data(), rowy.size() * 4, &p))) return rc;
        P.rowy = (const uint32_t*)p;
        if ((rc = dev_upload(t->dev_allocs, nullptr, (size_t)P.npanels * P.npiece * 8, &p))) return rc;
        P.piece = (uint64_t*)p;
        if (int e = launch_panel_pieces(s, P))
            return set_error(DQ_ECUDA, "panel pieces: %s", cudaGetErrorString((cudaError_t)e));
    }
    t->split = split;
    (warp ? t->pw_ok : t->panel_ok) = true;
    return DQ_OK;
}

int build_panel_plan(const dq_sector* s, double C, bool uniform_lin,
                     const std::vector<std::pair<std::pair<int, int>, std::pair<double, double>>>& pairs, dq_terms* t) {
    t->panel_ok = false;
    t->pw_ok = false;
    t->split = false;
    if (s->Q != 2 || s->n_sub < 2 || !uniform_lin || s->wide) return DQ_OK;
    bool fits = false;
    // the form dq_terms_path reports is the sector's own, whichever kernel runs
    bool own = false;
    if (int rc = build_form(s, C, pairs, t, false, true, &own)) return rc;
    const int ns = s->n_sub, last = s->Lk[ns - 1];
    const bool warp = last >= 8 && last <= 10, tail = ns >= 3 && !warp;
    const int own_sites = !own ? 0 : tail ? s->Lk[ns - 2] + last : last;
    if ((own || ns >= 3) && use_split_order(s, own_sites, own && !warp)) {
        if (int rc = build_form(s, C, pairs, t, true, true, &fits)) return rc;
        if (fits) {
            if (int rc = build_form(s, C, pairs, t, true, false, &fits)) return rc;
            if (!own) t->panel_ok = t->pw_ok = false;
            return DQ_OK;
        }
    }
    return build_form(s, C, pairs, t, false, false, &fits);
}

}  // namespace dq

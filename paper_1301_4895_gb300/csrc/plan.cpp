// Host side of the evaluation plans (plan.h): keys of a list's components,
// sink tensors, and the minor form of small point-sink lists.
#include "plan.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <new>

namespace mbc {

namespace {

int64_t binom_p(int n, int k) {
    if (k < 0 || k > n) return 0;
    int64_t r = 1;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return r;
}

uint32_t unrank(int64_t r, int k, int n) {
    uint32_t m = 0;
    for (int t = k; t >= 1; --t) {
        int p = t - 1;
        while (p + 1 < n && binom_p(p + 1, t) <= r) ++p;
        r -= binom_p(p, t);
        m |= 1u << p;
    }
    return m;
}

int parity(uint32_t x, uint32_t y) {
    int n = 0;
    for (; y; y &= y - 1) n += __builtin_popcount(x >> (__builtin_ctz(y) + 1));
    return n & 1;
}

bool disjoint(const PlanKey &a, const PlanKey &b) {
    return !(a.dp & b.dp) && !(a.dn & b.dn) && !(a.u & b.u) && !(a.d & b.d);
}

// key of a block component [spin][pair rank][single]
PlanKey block_key(int64_t i, int baryon, int nxi) {
    const int64_t npair = binom_p(nxi, 2);
    const uint32_t single = 1u << (i % nxi), pair = unrank((i / nxi) % npair, 2, nxi);
    const uint32_t spin = 1u << (i / nxi / npair);
    return baryon == MBC_PROTON ? PlanKey{spin, 0, pair, single} : PlanKey{0, spin, single, pair};
}

// key of component z of stage m (1-based); false if the operations disagree
bool stage_key(const mbc_term_list &L, int m, int64_t z, PlanKey &key) {
    if (m == 1) {
        if (z < 0 || z >= L.block_size) return false;
        key = block_key(z, L.path[0], L.nxi);
        return true;
    }
    const Step &s = L.steps[(size_t)m - 2];
    if (z < 0 || z >= s.n_z) return false;
    if (s.generated) {
        int64_t i = s.zrank.empty() ? z : s.zrank[(size_t)z];
        const int n[4] = {L.dim_snk, L.dim_snk, L.nxi, L.nxi};
        uint32_t v[4];
        for (int g = 3; g >= 0; --g) {
            const int64_t radix = binom_p(n[g], s.zk[g]);
            if (radix < 1) return false;
            v[g] = unrank(i % radix, s.zk[g], n[g]);
            i /= radix;
        }
        key = {v[0], v[1], v[2], v[3]};
        return true;
    }
    if (s.k < 1) return false;
    const size_t o = (size_t)(z * s.k);
    PlanKey x;
    if (!stage_key(L, m - 1, s.x[o], x)) return false;
    const PlanKey y = block_key(s.ys[o] & 0x7fff, s.baryon, L.nxi);
    if (!disjoint(x, y)) return false;
    key = {x.dp | y.dp, x.dn | y.dn, x.u | y.u, x.d | y.d};
    return true;
}

}  // namespace

bool list_entries(const mbc_term_list &L, std::vector<std::vector<PlanEntry>> &comp) {
    comp.assign((size_t)L.n_comp, {});
    if (L.pauli_forbidden || (int)L.steps.size() != L.A - 1) return false;
    for (double l : L.fin_l)
        if (!std::isfinite(l)) return false;  // plans compare and merge equal values
    for (const auto &pt : L.parts) {
        if (pt.A < 1 || pt.A > L.A || pt.n_p < 0 || pt.n_n < 0 || pt.n_p + pt.n_n != pt.A) return false;
        for (int c = pt.c0; c < pt.c1; ++c)
            for (int64_t e = L.fin_off[(size_t)c]; e < L.fin_off[(size_t)c + 1]; ++e) {
                PlanKey z;
                if (!stage_key(L, pt.A, L.fin_z[(size_t)e], z)) return false;
                if (__builtin_popcount(z.dp) != pt.n_p || __builtin_popcount(z.dn) != pt.n_n ||
                    __builtin_popcount(z.u) != 2 * pt.n_p + pt.n_n || __builtin_popcount(z.d) != pt.n_p + 2 * pt.n_n)
                    return false;
                comp[(size_t)c].push_back({z, L.fin_l[(size_t)e]});
            }
    }
    return true;
}

bool complete_operations(const mbc_term_list &L) {
    if ((L.dim != 2 && L.dim != 4) || L.nxi != 3 * L.dim * L.n_sources || L.dim_snk != L.dim * L.n_sinks ||
        (int)L.steps.size() != L.A - 1 || L.A < 1)
        return false;
    std::vector<PlanKey> block[2], x;  // keys of the block (by species) and of the stage so far
    for (int b : {MBC_PROTON, MBC_NEUTRON})
        for (int64_t i = 0; i < L.block_size; ++i) block[b == MBC_NEUTRON].push_back(block_key(i, b, L.nxi));
    x = block[L.path[0] == MBC_NEUTRON];
    int n_p = L.path[0] != MBC_NEUTRON, n_n = 1 - n_p;
    for (const Step &s : L.steps) {
        const bool proton = s.baryon == MBC_PROTON;
        const int xk[4] = {n_p, n_n, 2 * n_p + n_n, n_p + 2 * n_n};
        (proton ? n_p : n_n) += 1;
        const int zk[4] = {n_p, n_n, 2 * n_p + n_n, n_p + 2 * n_n};
        if (s.k != binom_p(proton ? n_p : n_n, 1) * binom_p(zk[2], proton ? 2 : 1) * binom_p(zk[3], proton ? 1 : 2) ||
            (int64_t)x.size() != s.n_x)
            return false;
        std::vector<PlanKey> z((size_t)s.n_z);
        if (s.generated) {
            // regenerated from the key: complete where both stages are dense
            if (!s.zrank.empty() || !s.xmap.empty() || !std::equal(zk, zk + 4, s.zk) || !std::equal(xk, xk + 4, s.xk))
                return false;
            const int n[4] = {L.dim_snk, L.dim_snk, L.nxi, L.nxi};
            const int64_t radix[3] = {binom_p(n[1], zk[1]), binom_p(n[2], zk[2]), binom_p(n[3], zk[3])};
#pragma omp parallel for
            for (int64_t i = 0; i < s.n_z; ++i)
                z[(size_t)i] = {unrank(i / radix[2] / radix[1] / radix[0], zk[0], n[0]),
                                unrank(i / radix[2] / radix[1] % radix[0], zk[1], n[1]),
                                unrank(i / radix[2] % radix[1], zk[2], n[2]), unrank(i % radix[2], zk[3], n[3])};
        } else {
            std::atomic<bool> ok{true};
            const std::vector<PlanKey> &f = block[!proton];
#pragma omp parallel
            {
                std::vector<int64_t> seen;  // output whose operations name this block entry
                try {
                    seen.assign(f.size(), -1);
                } catch (const std::bad_alloc &) {
                    ok = false;
                }
#pragma omp for schedule(dynamic, 256)
                for (int64_t i = 0; i < s.n_z; ++i)
                    for (int64_t j = 0; ok && j < s.k; ++j) {
                        const size_t o = (size_t)(i * s.k + j);
                        const PlanKey &a = x[s.x[o]], &b = f[s.ys[o] & 0x7fff];
                        PlanKey &k = z[(size_t)i];
                        if (j == 0) {
                            k = {a.dp | b.dp, a.dn | b.dn, a.u | b.u, a.d | b.d};
                            if (__builtin_popcount(k.dp) != zk[0] || __builtin_popcount(k.dn) != zk[1] ||
                                __builtin_popcount(k.u) != zk[2] || __builtin_popcount(k.d) != zk[3])
                                ok = false;
                        }
                        const int neg = parity(a.dp, b.dp) ^ parity(a.dn, b.dn) ^ parity(a.u, b.u) ^ parity(a.d, b.d);
                        if (!disjoint(a, b) || (a.dp | b.dp) != k.dp || (a.dn | b.dn) != k.dn || (a.u | b.u) != k.u ||
                            (a.d | b.d) != k.d || seen[s.ys[o] & 0x7fff] == i || (s.ys[o] >> 15) != neg)
                            ok = false;
                        else
                            seen[s.ys[o] & 0x7fff] = i;
                    }
            }
            if (!ok) return false;
        }
        x.swap(z);
    }
    return true;
}

std::vector<SpeciesEntry> species_tensor(int dim, uint32_t spins) {
    static const int gamma2[4][3] = {{0, 1, -1}, {1, 0, 1}, {2, 3, -1}, {3, 2, 1}};  // C gamma_5
    static const int eps[6][4] = {{0, 1, 2, 1}, {1, 2, 0, 1}, {2, 0, 1, 1}, {0, 2, 1, -1}, {2, 1, 0, -1}, {1, 0, 2, -1}};
    std::vector<SpeciesEntry> cur{{0, 0, 1}};
    for (uint32_t m = spins; m; m &= m - 1) {
        const int a = __builtin_ctz(m);
        std::map<std::pair<uint32_t, uint32_t>, int64_t> next;
        for (int g = 0; g < dim; ++g)
            for (const auto &e : eps) {
                const int x1 = 3 * a + e[0], x2 = 3 * gamma2[g][0] + e[1], x3 = 3 * gamma2[g][1] + e[2];
                if (x1 == x2) continue;
                const uint32_t pair = (1u << x1) | (1u << x2), single = 1u << x3;
                const int64_t v = (int64_t)gamma2[g][2] * e[3] * (x1 < x2 ? 1 : -1);
                for (const auto &c : cur)
                    if (!(c.pair & pair) && !(c.single & single))
                        next[{c.pair | pair, c.single | single}] +=
                            c.v * v * ((parity(c.pair, pair) ^ parity(c.single, single)) ? -1 : 1);
            }
        cur.clear();
        for (const auto &n : next)
            if (n.second) cur.push_back({n.first.first, n.first.second, n.second});
    }
    return cur;
}

namespace {

// Minors of one site's tile wanted by a list, with the products that make
// them: order 2 from two tile entries, 4 from two order-2 minors of fixed row
// pairs, the others from one row and the next lower order.
struct MinorBuilder {
    int nxi;
    std::map<std::pair<uint32_t, uint32_t>, int> index[8];  // (rows, columns) -> entry
    explicit MinorBuilder(int n) : nxi(n) {}

    int want(uint32_t rows, uint32_t cols) {
        const int o = __builtin_popcount(rows);
        if (o == 1) return __builtin_ctz(rows) * nxi + __builtin_ctz(cols);
        auto &ix = index[o];
        auto it = ix.find({rows, cols});
        if (it != ix.end()) return it->second;
        const int id = (int)ix.size();
        ix[{rows, cols}] = id;
        return id;
    }
    static int split_order(int o) { return o == 4 ? 2 : 1; }

    // order by order from the highest: the operands of every wanted minor
    void finish(MinorPlan &P) {
        std::vector<MinorPlan::Step> down;
        for (int o = 7; o >= 2; --o) {
            if (index[o].empty()) continue;
            const int a = split_order(o);
            MinorPlan::Step s;
            s.x_reg = a;
            s.y_reg = o - a;
            s.z_reg = o;
            s.n_z = (int32_t)index[o].size();
            s.k = (int32_t)binom_p(o, a);
            std::vector<std::pair<uint32_t, uint32_t>> keys((size_t)s.n_z);
            for (const auto &e : index[o]) keys[(size_t)e.second] = e.first;
            for (const auto &key : keys) {
                uint32_t r = key.first;  // the a lowest rows are expanded along
                for (int i = 0; i < a; ++i) r &= r - 1;
                const uint32_t top = key.first ^ r;
                for (uint32_t c = (0u - key.second) & key.second; c; c = (c - key.second) & key.second) {
                    if (__builtin_popcount(c) != a) continue;
                    s.x.push_back((uint16_t)want(top, c));
                    s.y.push_back((uint16_t)want(r, key.second ^ c));
                    s.neg.push_back((uint8_t)parity(c, key.second ^ c));
                }
            }
            P.reg_size[o] = s.n_z;
            down.push_back(std::move(s));
        }
        P.reg_size[1] = nxi * nxi;
        P.steps.assign(down.rbegin(), down.rend());
    }
};

constexpr int64_t kMaxMinorTerms = 1 << 14;
constexpr int kMaxMinorRuns = 32;   // partial rows of the lanes-are-sites kernel
constexpr int kMaxMinorRows = 256;  // operand rows its packed words address

std::shared_ptr<const MinorPlan> make_minor_plan(const mbc_term_list &L) {
    if (L.dim != 2 || L.nxi != 6 || L.n_sources != 1 || L.n_sinks != 1 || L.n_comp < 1 || L.A > 4) return nullptr;
    std::vector<std::vector<PlanEntry>> comp;
    if (!list_entries(L, comp)) return nullptr;
    std::map<std::pair<uint32_t, uint32_t>, std::vector<SpeciesEntry>> sink;  // (U', D') as (pair, single)
    int64_t bound = 0;
    for (const auto &pt : L.parts)
        for (int c = pt.c0; c < pt.c1; ++c)
            for (const auto &e : comp[(size_t)c]) {
                auto &t = sink[{e.z.dp, e.z.dn}];
                if (t.empty()) {
                    // full signed sums: n_P! n_N! times the ordered product
                    const double orders = std::tgamma(pt.n_p + 1.0) * std::tgamma(pt.n_n + 1.0);
                    std::map<std::pair<uint32_t, uint32_t>, int64_t> sum;
                    for (const auto &p : species_tensor(L.dim, e.z.dp))
                        for (const auto &n : species_tensor(L.dim, e.z.dn)) {
                            if ((p.pair & n.single) || (p.single & n.pair)) continue;
                            const int neg = parity(p.pair, n.single) ^ parity(p.single, n.pair);
                            sum[{p.pair | n.single, p.single | n.pair}] += p.v * n.v * (neg ? -1 : 1) * (int64_t)orders;
                        }
                    for (const auto &s : sum)
                        if (s.second) t.push_back({s.first.first, s.first.second, s.second});
                }
                if ((bound += (int64_t)t.size()) > kMaxMinorTerms) return nullptr;
            }
    auto P = std::make_shared<MinorPlan>();
    MinorBuilder mb(L.nxi);
    P->run_off.push_back(0);
    P->term_off.push_back(0);
    for (const auto &pt : L.parts) {
        const int nu = 2 * pt.n_p + pt.n_n, nd = pt.n_p + 2 * pt.n_n;
        for (int c = pt.c0; c < pt.c1; ++c) {
            // product of minors -> coefficient; the tile is the same for both
            // flavours, so minors of equal order commute into one term
            std::map<std::pair<int, int>, double> coef;
            for (const auto &e : comp[(size_t)c])
                for (const auto &s : sink[{e.z.dp, e.z.dn}]) {
                    int a = mb.want(s.pair, e.z.u), b = mb.want(s.single, e.z.d);
                    if (nu == nd && a > b) std::swap(a, b);
                    coef[{a, b}] += e.l * (double)s.v;
                }
            std::map<double, std::vector<MinorPlan::Term>> runs;  // by magnitude
            for (const auto &t : coef)
                if (t.second != 0.0)
                    runs[std::fabs(t.second)].push_back({(uint8_t)nu, (uint8_t)nd, (uint16_t)t.first.first,
                                                         (uint16_t)t.first.second, t.second < 0.0});
            for (const auto &r : runs) {
                P->run_coef.push_back(r.first);
                P->terms.insert(P->terms.end(), r.second.begin(), r.second.end());
                P->term_off.push_back((int32_t)P->terms.size());
            }
            P->run_off.push_back((int32_t)P->run_coef.size());
        }
    }
    if ((int)P->run_off.size() != L.n_comp + 1 || (int)P->run_coef.size() > kMaxMinorRuns) return nullptr;
    mb.finish(*P);
    // complex multiply-adds per site of both forms: the list's own steps with
    // their blocks (diquark 3 nxi^2 of 4 terms, one species' block of 6 terms)
    int64_t minor = (int64_t)P->terms.size(), chain = 3LL * L.nxi * L.nxi * 4 + 6 * L.block_size;
    for (const auto &s : P->steps) {
        minor += (int64_t)s.n_z * s.k;
        if (s.n_z > kMaxMinorRows) return nullptr;
    }
    for (const auto &s : L.steps) chain += s.n_z * s.k;
    return minor < chain ? P : nullptr;
}

std::shared_ptr<const SaturatedPlan> make_saturated_plan(const mbc_term_list &L) {
    if (L.dim != 4 || L.n_sources != 1 || L.n_sinks != 1 || L.n_comp < 1 || L.parts.size() != 1) return nullptr;
    const auto &pt = L.parts[0];
    if (2 * pt.n_p + pt.n_n != L.nxi || pt.n_p + 2 * pt.n_n != L.nxi || pt.c0 != 0 || pt.c1 != L.n_comp) return nullptr;
    std::vector<std::vector<PlanEntry>> comp;
    if (!list_entries(L, comp)) return nullptr;
    const uint32_t all = (1u << L.nxi) - 1;
    auto P = std::make_shared<SaturatedPlan>();
    std::map<std::pair<uint32_t, uint32_t>, double> sink;
    for (const auto &entries : comp) {
        double v = 0.0;
        for (const auto &e : entries) {
            auto it = sink.find({e.z.dp, e.z.dn});
            if (it == sink.end()) {
                std::map<std::pair<uint32_t, uint32_t>, int64_t> neutron;
                for (const auto &n : species_tensor(L.dim, e.z.dn)) neutron[{n.single, n.pair}] = n.v;
                double t = 0.0;
                for (const auto &p : species_tensor(L.dim, e.z.dp)) {
                    const auto n = neutron.find({all ^ p.pair, all ^ p.single});
                    if (n == neutron.end()) continue;
                    const int neg = parity(p.pair, n->first.first) ^ parity(p.single, n->first.second);
                    t += (double)p.v * (double)n->second * (neg ? -1.0 : 1.0);
                }
                // full signed sums: n_P! n_N! times the ordered product
                t *= std::tgamma(pt.n_p + 1.0) * std::tgamma(pt.n_n + 1.0);
                it = sink.insert({{e.z.dp, e.z.dn}, t}).first;
            }
            v += e.l * it->second;
        }
        P->coef.push_back(v / pt.norm);
    }
    return P;
}

int64_t rank_of(uint32_t m) {
    int64_t r = 0;
    for (int t = 1; m; m &= m - 1, ++t) r += binom_p(__builtin_ctz(m), t);
    return r;
}

// (subset, rest, sign of subset | rest) for every k-subset of a set
struct Split {
    uint32_t sub, rest;
    int neg;
};
std::vector<Split> splits_of(uint32_t set, int k) {
    std::vector<Split> out;
    for (uint32_t c = (0u - set) & set; c; c = (c - set) & set)
        if (__builtin_popcount(c) == k) out.push_back({c, set ^ c, parity(c, set ^ c)});
    return out;
}

struct PairEntry {
    uint32_t i, j;
    double v;
};
// Rows of one group's matrix: [0] P rows gathering N, [1] N rows gathering P.
struct PairRows {
    struct Row {
        uint32_t id;
        int64_t e0, e1;
        int32_t block;
        uint16_t cls;
    };
    std::vector<Row> rows[2];
    std::vector<uint32_t> col;
    std::vector<double> val;
};

// Assign every entry to its P row or its N row by a greedy vertex cover (the
// vertex with the most unassigned entries next) and order the rows by
// connected block, then by their columns. n_n = 0: one vertex set for both
// sides (symmetric matrix), P rows only.
template <class ClassOf>
void pair_rows(const std::vector<PairEntry> &all, int64_t n_p, int64_t n_n, ClassOf &&class_of, PairRows &R) {
    const bool sym = n_n == 0;
    const size_t nv = (size_t)(n_p + n_n);
    auto vert = [&](const PairEntry &e, int s) { return s == 0 || sym ? (s ? e.j : e.i) : (uint32_t)(n_p + e.j); };
    std::vector<int64_t> off(nv + 1, 0);
    std::vector<int32_t> up(nv);
    for (size_t v = 0; v < nv; ++v) up[v] = (int32_t)v;
    auto find = [&](uint32_t v) {
        while (up[v] != (int32_t)v) v = (uint32_t)(up[v] = up[(size_t)up[v]]);
        return v;
    };
    for (const auto &e : all) {
        const uint32_t a = vert(e, 0), b = vert(e, 1);
        ++off[a + 1];
        if (b != a) ++off[b + 1];
        const uint32_t x = find(a), y = find(b);
        if (x != y) up[std::max(x, y)] = (int32_t)std::min(x, y);
    }
    for (size_t v = 0; v < nv; ++v) off[v + 1] += off[v];
    std::vector<int64_t> at(off.begin(), off.end() - 1), deg(nv);
    std::vector<int32_t> adj((size_t)off[nv]);
    for (size_t k = 0; k < all.size(); ++k) {
        const uint32_t a = vert(all[k], 0), b = vert(all[k], 1);
        adj[(size_t)at[a]++] = (int32_t)k;
        if (b != a) adj[(size_t)at[b]++] = (int32_t)k;
    }
    std::vector<uint8_t> taken(all.size(), 0);
    std::vector<std::vector<uint32_t>> bucket;
    for (size_t v = 0; v < nv; ++v) {
        deg[v] = off[v + 1] - off[v];
        if (deg[v] >= (int64_t)bucket.size()) bucket.resize((size_t)deg[v] + 1);
        if (deg[v]) bucket[(size_t)deg[v]].push_back((uint32_t)v);
    }
    R.col.reserve(all.size());
    R.val.reserve(all.size());
    for (int64_t d = (int64_t)bucket.size() - 1; d > 0; --d)
        for (size_t q = 0; q < bucket[(size_t)d].size(); ++q) {
            const uint32_t v = bucket[(size_t)d][q];
            if (deg[v] != d) {  // lost entries since it was filed
                if (deg[v] > 0 && deg[v] < d) bucket[(size_t)deg[v]].push_back(v);
                continue;
            }
            const bool n_row = !sym && (int64_t)v >= n_p;
            PairRows::Row row{n_row ? (uint32_t)(v - n_p) : v, (int64_t)R.col.size(), 0, (int32_t)find(v), 0};
            row.cls = class_of(row.id, n_row ? 1 : 0);
            std::vector<std::pair<uint32_t, double>> entries;
            for (int64_t k = off[v]; k < off[v + 1]; ++k) {
                const int32_t e = adj[(size_t)k];
                if (taken[(size_t)e]) continue;
                taken[(size_t)e] = 1;
                const uint32_t a = vert(all[(size_t)e], 0), b = vert(all[(size_t)e], 1), o = a == v ? b : a;
                entries.push_back({n_row || sym ? o : all[(size_t)e].j, all[(size_t)e].v});
                if (o != v) --deg[o];
            }
            deg[v] = 0;
            std::sort(entries.begin(), entries.end());
            for (const auto &e : entries) {
                R.col.push_back(e.first);
                R.val.push_back(e.second);
            }
            row.e1 = (int64_t)R.col.size();
            R.rows[n_row ? 1 : 0].push_back(row);
        }
    for (auto &rows : R.rows)
        std::sort(rows.begin(), rows.end(), [&](const PairRows::Row &a, const PairRows::Row &b) {
            if (a.cls != b.cls) return a.cls < b.cls;
            if (a.block != b.block) return a.block < b.block;
            return std::lexicographical_compare(R.col.begin() + a.e0, R.col.begin() + a.e1, R.col.begin() + b.e0,
                                                R.col.begin() + b.e1);
        });
}

// Runs of one range's rows (quark sets of four): the triple that most of the
// remaining sets contain, up to kProdRun of them, and so on - the longest first.
bool prod_runs(const std::vector<uint32_t> &sets, int nxi, PairPlan &P) {
    if (sets.size() > 512) return false;  // a record's row field; C(12, 4) = 495
    std::vector<uint8_t> done(sets.size(), 0);
    std::vector<int> count((size_t)1 << nxi);
    for (size_t left = sets.size(); left > 0;) {
        std::fill(count.begin(), count.end(), 0);
        uint32_t triple = 0;
        for (size_t r = 0; r < sets.size(); ++r)
            for (uint32_t s = done[r] ? 0u : sets[r]; s; s &= s - 1) {
                const uint32_t t = sets[r] ^ (s & (0u - s));
                if (++count[t] > (triple ? count[triple] : 0)) triple = t;
            }
        const uint32_t a = triple & (0u - triple), c = 1u << (31 - __builtin_clz(triple)), b = triple ^ a ^ c;
        const uint32_t held[3] = {a | b, a | c, b | c};
        PairPlan::ProdRun run{(uint32_t)P.prod_rec.size(), 0, {}};
        for (int k = 0; k < 3; ++k) run.pair[k] = (uint8_t)rank_of(held[k]);
        for (size_t r = 0; r < sets.size() && run.n < PairPlan::kProdRun; ++r) {
            if (done[r] || (sets[r] & triple) != triple) continue;
            uint32_t rec = (uint32_t)r << 21, odd = 3;
            for (int k = 0; k < 3; ++k) {
                const uint32_t other = sets[r] ^ held[k];
                rec |= (uint32_t)rank_of(other) << (7 * k);
                if (parity(held[k], other)) odd = odd == 3 ? (uint32_t)k : 4u;
            }
            if (odd > 2) return false;  // one of the three splits interleaves
            P.prod_rec.push_back(rec | odd << 30);
            done[r] = 1;
            ++run.n;
            --left;
        }
        P.prod_runs.push_back(run);
    }
    return true;
}

constexpr int64_t kMaxPairEntries = (int64_t)1 << 26;  // 12 B each on the device

std::shared_ptr<const PairPlan> make_pair_plan(const mbc_term_list &L) {
    if (L.parts.size() != 1 || L.nxi > 12 || L.n_comp < 1) return nullptr;
    const auto &pt = L.parts[0];
    const int np = pt.n_p, nn = pt.n_n, nxi = L.nxi;
    if (np < 1 || np > 2 || nn < 1 || nn > 2 || pt.c0 != 0 || pt.c1 != L.n_comp) return nullptr;
    for (const auto &s : L.steps)
        if (s.generated) return nullptr;  // list-free lists keep no tables
    std::vector<std::vector<PlanEntry>> comp;
    if (!list_entries(L, comp)) return nullptr;
    // evaluations: (sink spin sets, tensor), the tensor a list of (U, D, l) in
    // key order (the list's contraction entries are sorted by key)
    using UD = std::pair<uint32_t, uint32_t>;
    using Tensor = std::vector<std::pair<UD, double>>;
    struct Group {
        Tensor t;
        bool sym = false;
        std::map<uint32_t, int> mp, mn;  // spin sets -> position
    };
    std::map<Tensor, int> ids;
    std::vector<Group> groups;
    struct Eval {
        int group;
        uint32_t dp, dn;
    };
    auto exchanged = [](const Tensor &t) {
        Tensor x;
        x.reserve(t.size());
        for (const auto &e : t) x.push_back({{e.first.second, e.first.first}, e.second});
        std::sort(x.begin(), x.end());
        return x;
    };
    std::vector<std::vector<Eval>> evals((size_t)L.n_comp);
    for (int c = 0; c < L.n_comp; ++c) {
        std::map<UD, Tensor> by_sink;
        for (const auto &e : comp[(size_t)c])
            if (e.l != 0.0) by_sink[{e.z.dp, e.z.dn}].push_back({{e.z.u, e.z.d}, e.l});
        std::vector<PlanEntry>().swap(comp[(size_t)c]);
        for (auto &sk : by_sink) {
            uint32_t dp = sk.first.first, dn = sk.first.second;
            std::sort(sk.second.begin(), sk.second.end());
            auto it = ids.find(sk.second);
            if (it == ids.end() && np == nn) {  // of the two flavour-exchanged forms the first one seen
                Tensor ex = exchanged(sk.second);
                it = ids.find(ex);
                if (it != ids.end())
                    std::swap(dp, dn);
                else if (ex == sk.second)
                    groups.push_back({{}, true, {}, {}});
            }
            if (it == ids.end()) {
                if (groups.size() == ids.size()) groups.push_back({});
                it = ids.insert({sk.second, (int)ids.size()}).first;
                groups.back().t = sk.second;
            }
            const int g = it->second;
            groups[(size_t)g].mp[dp] = groups[(size_t)g].mn[dn] = 0;
            evals[(size_t)c].push_back({g, dp, dn});
        }
    }
    ids.clear();
    int64_t total = 0;
    const int64_t per_z = binom_p(2 * np + nn, 2 * np) * binom_p(np + 2 * nn, np);
    for (auto &g : groups) {
        total += (int64_t)g.t.size() * per_z;
        if (g.sym) {  // both orders of a pair of sets are evaluated
            g.mp.insert(g.mn.begin(), g.mn.end());
            g.mn = g.mp;
        }
    }
    if (total > kMaxPairEntries) return nullptr;
    auto P = std::make_shared<PairPlan>();
    P->np = np;
    P->nn = nn;
    // rows: block entries [pair][single] for one baryon; for two the (4-set,
    // 2-set) keys some entry names, 2-set slowest
    const int64_t nset2 = binom_p(nxi, 2), nset4 = binom_p(nxi, 4), wide = nset4 * nset2;
    const int64_t n_of[2] = {np == 2 ? wide : nset2 * nxi, nn == 2 ? wide : nset2 * nxi};
    std::vector<int32_t> row_of((size_t)((np == 2 || nn == 2) ? wide : 0), -1);
    auto full_row = [&](uint32_t pair, uint32_t single, int n) {
        return n == 2 ? rank_of(single) * nset4 + rank_of(pair) : rank_of(pair) * nxi + rank_of(single);
    };
    // colour content of a full row: how many of its quarks have colours 0 and 1
    std::vector<uint16_t> cls[2];
    for (int s = 0; s < 2; ++s) {
        const int n = s ? nn : np;
        if (s == 1 && nn == np) {
            cls[1] = cls[0];
            break;
        }
        auto colours = [&](uint32_t m) {
            uint16_t v = 0;
            for (; m; m &= m - 1) {
                const int col = (__builtin_ctz(m) / L.n_sources) % 3;
                v = (uint16_t)(v + (col == 0 ? 16 : col == 1 ? 1 : 0));
            }
            return v;
        };
        const int64_t second = n == 2 ? nset4 : nxi;  // fastest index: 4-set or single
        std::vector<uint16_t> slow, fast;
        for (int64_t r = 0; r < n_of[s] / second; ++r) slow.push_back(colours(unrank(r, 2, nxi)));
        for (int64_t r = 0; r < second; ++r) fast.push_back(colours(unrank(r, n == 2 ? 4 : 1, nxi)));
        for (int64_t r = 0; r < n_of[s]; ++r)
            cls[s].push_back((uint16_t)(slow[(size_t)(r / second)] + fast[(size_t)(r % second)]));
    }
    auto class_of = [&](uint32_t row, int side) { return cls[side][row]; };
    std::vector<PairRows> lam(groups.size());
    std::atomic<bool> failed{false};
#pragma omp parallel for schedule(dynamic, 1)
    for (size_t g = 0; g < groups.size(); ++g) {
        try {
            std::vector<PairEntry> all;
            all.reserve(groups[g].t.size() * (size_t)per_z);
            std::map<uint32_t, std::vector<Split>> us, ds;
            for (const auto &t : groups[g].t) {
                const double l = t.second;
                auto &u = us[t.first.first], &d = ds[t.first.second];
                if (u.empty()) u = splits_of(t.first.first, 2 * np);
                if (d.empty()) d = splits_of(t.first.second, np);
                for (const auto &a : u)
                    for (const auto &e : d) {
                        const uint32_t i = (uint32_t)full_row(a.sub, e.sub, np), j = (uint32_t)full_row(e.rest, a.rest, nn);
                        const double v = (a.neg ^ e.neg) ? -l : l;
                        if (!groups[g].sym || i < j)
                            all.push_back({i, j, v});
                        else if (i == j)
                            all.push_back({i, j, 0.5 * v});
                    }
            }
            pair_rows(all, n_of[0], groups[g].sym ? 0 : n_of[1], class_of, lam[g]);
        } catch (const std::bad_alloc &) {
            failed = true;
        }
    }
    if (failed) throw std::bad_alloc();
    const int n_side[2] = {np, nn};
    for (const auto &R : lam)
        for (int s = 0; s < 2; ++s) {
            const auto &rows = R.rows[s];
            for (const auto &r : rows) {
                if (n_side[s] == 2) row_of[r.id] = 0;
                for (int64_t e = r.e0; e < r.e1; ++e) {
                    if (n_side[1 - s] == 2) row_of[R.col[(size_t)e]] = 0;
                    P->val_fp32 = P->val_fp32 && (double)(float)R.val[(size_t)e] == R.val[(size_t)e];
                }
            }
        }
    std::vector<UD> rows2;
    for (int64_t r = 0; r < (int64_t)row_of.size(); ++r)
        if (row_of[(size_t)r] == 0) {
            row_of[(size_t)r] = P->n_rows2++;
            rows2.push_back({unrank(r % nset4, 4, nxi), unrank(r / nset4, 2, nxi)});
        }
    // elements: spin values for one baryon, used two-spin sets for two
    std::map<uint32_t, int32_t> elem2;
    for (const auto &g : groups) {
        if (np == 2)
            for (const auto &m : g.mp) elem2[m.first] = 0;
        if (nn == 2)
            for (const auto &m : g.mn) elem2[m.first] = 0;
    }
    for (auto &m : elem2) {
        m.second = (int32_t)P->masks2.size();
        P->masks2.push_back(m.first);
    }
    auto elem = [&](uint32_t mask, int n) { return n == 2 ? elem2[mask] : (int32_t)__builtin_ctz(mask); };
    int64_t work = 0;
    P->row_ptr.push_back(0);
    for (size_t g = 0; g < groups.size(); ++g) {
        PairPlan::Group G;
        const int64_t nnz0 = (int64_t)P->col.size(), rows0 = (int64_t)P->row_id.size();
        for (int s = 0; s < 2; ++s) {
            G.row0[s] = (int64_t)P->row_id.size();
            for (const auto &r : lam[g].rows[s])
                for (int64_t e0 = r.e0; e0 < r.e1; e0 += kPackCols) {  // a longer row goes in pieces
                    for (int64_t e = e0; e < std::min(r.e1, e0 + kPackCols); ++e) {
                        const uint32_t j = lam[g].col[(size_t)e];
                        P->col.push_back(n_side[1 - s] == 2 ? (uint32_t)row_of[j] : j);
                        P->val.push_back(lam[g].val[(size_t)e]);
                    }
                    P->row_class.push_back(r.cls);
                    P->row_id.push_back(n_side[s] == 2 ? (uint32_t)row_of[r.id] : r.id);
                    P->row_ptr.push_back((int64_t)P->col.size());
                }
            G.row1[s] = (int64_t)P->row_id.size();
        }
        lam[g] = PairRows();
        for (auto &m : groups[g].mp) {
            m.second = (int)G.mp.size();
            G.mp.push_back(elem(m.first, np));
        }
        for (auto &m : groups[g].mn) {
            m.second = (int)G.mn.size();
            G.mn.push_back(elem(m.first, nn));
        }
        G.eval0 = P->n_evals;
        P->n_evals += (int64_t)(G.mp.size() * G.mn.size());
        work += ((int64_t)P->col.size() - nnz0) * (int64_t)G.mn.size() / 2 +
                ((int64_t)P->row_id.size() - rows0) * (int64_t)(G.mp.size() * G.mn.size());
        P->groups.push_back(std::move(G));
    }
    if (P->n_evals > (int64_t)1 << 20) return nullptr;
    work += 12LL * (int64_t)P->masks2.size() * P->n_rows2;
    // complex multiply-adds of the list's own recursion; both forms share blocks
    int64_t chain = 0;
    for (const auto &s : L.steps) chain += s.n_z * s.k;
    if (work * 5 > chain * 4) return nullptr;
    P->comp_off.push_back(0);
    for (int c = 0; c < L.n_comp; ++c) {
        for (const auto &e : evals[(size_t)c]) {
            const auto &g = groups[(size_t)e.group];
            const auto &G = P->groups[(size_t)e.group];
            auto ev = [&](uint32_t a, uint32_t b) {
                return (int32_t)(G.eval0 + (int64_t)g.mp.at(a) * (int64_t)G.mn.size() + g.mn.at(b));
            };
            P->comp_eval.push_back(ev(e.dp, e.dn));
            if (g.sym) P->comp_eval.push_back(ev(e.dn, e.dp));
        }
        P->comp_off.push_back((int32_t)P->comp_eval.size());
    }
    P->scale = std::tgamma(np + 1.0) * std::tgamma(nn + 1.0) / pt.norm;
    for (size_t r0 = 0, r1; r0 < rows2.size(); r0 = r1) {
        const uint32_t e = rows2[r0].second;
        for (r1 = r0; r1 < rows2.size() && rows2[r1].second == e;) ++r1;
        P->range_off.push_back((int32_t)r0);
        P->range_e.push_back((uint16_t)(__builtin_ctz(e) | __builtin_ctz(e & (e - 1)) << 8));
        std::vector<uint32_t> sets;
        for (size_t r = r0; r < r1; ++r) sets.push_back(rows2[r].first);
        P->run_off.push_back((int32_t)P->prod_runs.size());
        if (!prod_runs(sets, nxi, *P)) return nullptr;
    }
    if (!rows2.empty()) {
        P->range_off.push_back((int32_t)rows2.size());
        P->run_off.push_back((int32_t)P->prod_runs.size());
    }
    return P;
}

}  // namespace

namespace {
// A plan stands in for the list's operations, so those of a file must be the
// recursion's own, all of them (caller holds plan_mu).
template <class P>
std::shared_ptr<const P> replaces_ops(mbc_term_list *L, std::shared_ptr<const P> plan) {
    if (!plan || !L->from_file) return plan;
    if (!L->ops_checked) {
        L->ops_complete = complete_operations(*L);
        L->ops_checked = true;
    }
    return L->ops_complete ? plan : nullptr;
}
}  // namespace

std::shared_ptr<const PairPlan> pair_plan(const mbc_term_list *Lc) {
    mbc_term_list *L = const_cast<mbc_term_list *>(Lc);
    std::lock_guard<std::mutex> g(L->plan_mu);
    if (!L->pair_tried) {
        try {
            L->pair = replaces_ops(L, make_pair_plan(*L));
            L->pair_tried = true;
        } catch (const std::bad_alloc &) {
            return nullptr;
        }
    }
    return L->pair;
}

std::shared_ptr<const SaturatedPlan> saturated_plan(const mbc_term_list *Lc) {
    mbc_term_list *L = const_cast<mbc_term_list *>(Lc);
    std::lock_guard<std::mutex> g(L->plan_mu);
    if (!L->saturated_tried) {
        try {
            L->saturated = replaces_ops(L, make_saturated_plan(*L));
            L->saturated_tried = true;
        } catch (const std::bad_alloc &) {
            return nullptr;
        }
    }
    return L->saturated;
}

namespace {

std::shared_ptr<const MirrorPlan> make_mirror_plan(const mbc_term_list &L) {
    if (L.pauli_forbidden || L.A != 2 || L.parts.size() != 1 || L.parts[0].n_p != 1 || L.parts[0].n_n != 1 ||
        L.parts[0].A != 2 || L.steps.size() != 1 || L.steps[0].generated || L.steps[0].n_z >= 65536)
        return nullptr;
    auto P = std::make_shared<MirrorPlan>();
    std::map<std::vector<uint32_t>, int32_t> at;
    for (int64_t z = 0; z < L.steps[0].n_z; ++z) {
        PlanKey k;
        if (!stage_key(L, 2, z, k)) return nullptr;
        const auto m = at.find({k.dn, k.dp, k.d, k.u});
        if (m != at.end()) {
            P->rep.push_back(m->second);
            continue;
        }
        at[{k.dp, k.dn, k.u, k.d}] = (int32_t)P->keep.size();
        P->rep.push_back((int32_t)P->keep.size());
        P->keep.push_back((int32_t)z);
    }
    return P;
}

}  // namespace

std::shared_ptr<const MirrorPlan> mirror_plan(const mbc_term_list *Lc) {
    mbc_term_list *L = const_cast<mbc_term_list *>(Lc);
    std::lock_guard<std::mutex> g(L->plan_mu);
    if (!L->mirror_tried) {
        try {
            L->mirror = replaces_ops(L, make_mirror_plan(*L));
            L->mirror_tried = true;
        } catch (const std::bad_alloc &) {
            return nullptr;
        }
    }
    return L->mirror;
}

std::shared_ptr<const MinorPlan> minor_plan(const mbc_term_list *Lc) {
    mbc_term_list *L = const_cast<mbc_term_list *>(Lc);
    std::lock_guard<std::mutex> g(L->plan_mu);
    if (!L->minor_tried) {
        try {
            L->minor = replaces_ops(L, make_minor_plan(*L));
            L->minor_tried = true;
        } catch (const std::bad_alloc &) {
            return nullptr;  // the list's own operations serve; tried again at the next use
        }
    }
    return L->minor;
}

}  // namespace mbc

// Host side of the evaluation plans (plan.h): keys of a list's components,
// sink tensors, and the minor form of small point-sink lists.
#include "plan.h"

#include <algorithm>
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

}  // namespace

std::shared_ptr<const SaturatedPlan> saturated_plan(const mbc_term_list *Lc) {
    mbc_term_list *L = const_cast<mbc_term_list *>(Lc);
    std::lock_guard<std::mutex> g(L->plan_mu);
    if (!L->saturated_tried) {
        try {
            L->saturated = make_saturated_plan(*L);
            L->saturated_tried = true;
        } catch (const std::bad_alloc &) {
            return nullptr;
        }
    }
    return L->saturated;
}

std::shared_ptr<const MinorPlan> minor_plan(const mbc_term_list *Lc) {
    mbc_term_list *L = const_cast<mbc_term_list *>(Lc);
    std::lock_guard<std::mutex> g(L->plan_mu);
    if (!L->minor_tried) {
        try {
            L->minor = make_minor_plan(*L);
            L->minor_tried = true;
        } catch (const std::bad_alloc &) {
            return nullptr;  // the list's own operations serve; tried again at the next use
        }
    }
    return L->minor;
}

}  // namespace mbc

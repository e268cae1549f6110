// Host check of the evaluation plans (plan.h): on random propagators the minor
// form of a list gives the components that the list's own recursion gives,
// with every operand inside its region.
#include <complex>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "../../paper_1301_4895_gb300/csrc/builder.cpp"
#include "../../paper_1301_4895_gb300/csrc/plan.cpp"

namespace mbc {
void free_device_cache(mbc_term_list *) {}
}  // namespace mbc

using cd = std::complex<double>;

// blocks [spin][pair][single] of a tile S[row][col] (u = d: one block for both species)
static std::vector<cd> block(const mbc_term_list &L, const std::vector<cd> &S) {
    const int n = L.nxi, ns = L.n_sources;
    const int g2[4][3] = {{0, 1, -1}, {1, 0, 1}, {2, 3, -1}, {3, 2, 1}};
    auto lc = [](int a, int b, int c) { return (a - b) * (b - c) * (c - a) / 2; };
    (void)ns;
    std::vector<cd> f;
    for (int a = 0; a < L.dim; ++a)
        for (int j = 1; j < n; ++j)
            for (int i = 0; i < j; ++i)
                for (int s = 0; s < n; ++s) {
                    cd v = 0;
                    for (int g = 0; g < L.dim; ++g)
                        for (int c1 = 0; c1 < 3; ++c1)
                            for (int c2 = 0; c2 < 3; ++c2)
                                for (int c3 = 0; c3 < 3; ++c3) {
                                    const double e = lc(c1, c2, c3) * g2[g][2];
                                    if (e == 0) continue;
                                    const cd *r1 = &S[(size_t)(3 * a + c1) * n], *r2 = &S[(size_t)(3 * g2[g][0] + c2) * n],
                                             *r3 = &S[(size_t)(3 * g2[g][1] + c3) * n];
                                    v += e * (r1[i] * r2[j] - r1[j] * r2[i]) * r3[s];
                                }
                    f.push_back(v);
                }
    return f;
}

// components and their magnitudes by the list's own operations
static void chain(const mbc_term_list &L, const std::vector<cd> &f, std::vector<cd> &C, std::vector<double> &mag) {
    C.assign((size_t)L.n_comp, 0);
    mag.assign((size_t)L.n_comp, 0);
    std::vector<cd> x = f;
    for (int m = 1; m <= L.A; ++m) {
        if (m > 1) {
            const auto &s = L.steps[(size_t)m - 2];
            std::vector<cd> z((size_t)s.n_z, 0);
            for (int64_t i = 0; i < s.n_z; ++i)
                for (int64_t j = 0; j < s.k; ++j) {
                    const size_t o = (size_t)(i * s.k + j);
                    const cd t = x[s.x[o]] * f[s.ys[o] & 0x7fff];
                    z[(size_t)i] += s.ys[o] & 0x8000 ? -t : t;
                }
            x.swap(z);
        }
        for (const auto &pt : L.parts)
            for (int c = pt.c0; pt.A == m && c < pt.c1; ++c)
                for (int64_t e = L.fin_off[(size_t)c]; e < L.fin_off[(size_t)c + 1]; ++e) {
                    const cd t = L.fin_l[(size_t)e] * x[L.fin_z[(size_t)e]];
                    C[(size_t)c] += t;
                    mag[(size_t)c] += std::abs(t);
                }
    }
}

static int bad_minors(const char *name, const mbc_term_list &L, bool expect, std::mt19937 &rng) {
    const auto P = mbc::minor_plan(&L);
    if (!!P != expect) {
        std::printf("%s: minor form %s\n", name, P ? "made" : "not made");
        return 1;
    }
    if (!P) return 0;
    std::normal_distribution<double> nd;
    std::vector<cd> S((size_t)L.nxi * L.nxi);
    for (auto &v : S) v = cd(nd(rng), nd(rng));
    std::vector<cd> C;
    std::vector<double> mag;
    chain(L, block(L, S), C, mag);
    std::vector<cd> reg[8];
    reg[1] = S;
    for (const auto &s : P->steps) {
        reg[s.z_reg].assign((size_t)s.n_z, 0);
        for (int64_t o = 0; o < (int64_t)s.n_z * s.k; ++o) {
            const cd t = reg[s.x_reg].at(s.x[(size_t)o]) * reg[s.y_reg].at(s.y[(size_t)o]);
            reg[s.z_reg][(size_t)(o / s.k)] += s.neg[(size_t)o] ? -t : t;
        }
    }
    double worst = 0;
    for (int c = 0; c < L.n_comp; ++c) {
        cd v = 0;
        for (int r = P->run_off[(size_t)c]; r < P->run_off[(size_t)c + 1]; ++r)
            for (int e = P->term_off[(size_t)r]; e < P->term_off[(size_t)r + 1]; ++e) {
                const auto &t = P->terms[(size_t)e];
                const cd p = reg[t.x_reg].at(t.x) * reg[t.y_reg].at(t.y);
                v += (t.neg ? -1.0 : 1.0) * P->run_coef[(size_t)r] * p;
            }
        const double scale = mag[(size_t)c] > 0 ? mag[(size_t)c] : 1.0;
        worst = std::max(worst, std::abs(v - C[(size_t)c]) / scale);
    }
    std::printf("%s: minor form, %zu products, worst difference %.1e\n", name, P->terms.size(), worst);
    return worst > 1e-11;
}

static int bad_pairs(const char *name, const mbc_term_list &L, bool expect, std::mt19937 &rng) {
    const auto P = mbc::pair_plan(&L);
    if (!!P != expect) {
        std::printf("%s: pair form %s\n", name, P ? "made" : "not made");
        return 1;
    }
    if (!P) return 0;
    // any blocks will do: projected blocks are sums of blocks over sites
    std::normal_distribution<double> nd;
    std::vector<cd> f((size_t)L.block_size);
    for (auto &v : f) v = cd(nd(rng), nd(rng));
    std::vector<cd> C, prod;
    std::vector<double> mag;
    chain(L, f, C, mag);
    for (size_t r = 0; r < P->row_id.size(); ++r)
        if (P->row_ptr[r + 1] - P->row_ptr[r] > mbc::kPackCols) return 1;
    const int64_t npair = (int64_t)L.nxi * (L.nxi - 1) / 2;
    for (uint32_t m : P->masks2) {
        const int s1 = __builtin_ctz(m), s2 = __builtin_ctz(m & (m - 1));
        const size_t base = prod.size();
        prod.resize(base + (size_t)P->n_rows2, cd(NAN, NAN));  // every row is written
        for (size_t k = 0; k + 1 < P->range_off.size(); ++k)
            for (int u = P->run_off[k]; u < P->run_off[k + 1]; ++u) {
                const int e[2] = {P->range_e[k] & 255, P->range_e[k] >> 8};
                const auto &run = P->prod_runs.at((size_t)u);
                if (run.n < 1 || run.n > mbc::PairPlan::kProdRun) return 1;
                for (int t = 0; t < run.n; ++t) {
                    const uint32_t rec = P->prod_rec.at(run.rec0 + (size_t)t);
                    const int row = P->range_off[k] + (int)(rec >> 21 & 511);
                    if (row >= P->range_off[k + 1]) return 1;
                    cd v = 0;
                    for (int q = 0; q < 3; ++q)
                        for (int i = 0; i < 2; ++i) {
                            const int64_t held = run.pair[q], other = rec >> (7 * q) & 127;
                            if (held >= npair || other >= npair) return 1;
                            auto F = [&](int s, int64_t p, int j) { return f.at((size_t)((s * npair + p) * L.nxi + e[j])); };
                            const cd w = F(s1, held, i) * F(s2, other, 1 - i) + F(s1, other, i) * F(s2, held, 1 - i);
                            v += (rec >> 30 == (uint32_t)q) != (i == 1) ? -w : w;
                        }
                    prod[base + (size_t)row] = v;
                }
            }
    }
    const int64_t brows = L.block_size / L.dim_snk;
    const int64_t pr = P->p_rows(brows), nr = P->n_rows(brows);
    std::vector<cd> ev((size_t)P->n_evals, 0);
    // rows of side 0 gather neutron products, rows of side 1 proton products
    const std::vector<cd> &pv = P->np == 2 ? prod : f, &nv = P->nn == 2 ? prod : f;
    for (const auto &g : P->groups)
        for (int side = 0; side < 2; ++side)
            for (int64_t r = g.row0[side]; r < g.row1[side]; ++r) {
                const auto &rows = side ? g.mn : g.mp, &cols = side ? g.mp : g.mn;
                const std::vector<cd> &rv = side ? nv : pv, &cv = side ? pv : nv;
                const int64_t n_row = side ? nr : pr, n_col = side ? pr : nr;
                if (P->row_id[(size_t)r] >= n_row) return 1;
                for (size_t b = 0; b < cols.size(); ++b) {
                    cd y = 0;
                    for (int64_t e = P->row_ptr[(size_t)r]; e < P->row_ptr[(size_t)r + 1]; ++e) {
                        if (P->col[(size_t)e] >= n_col) return 1;
                        y += P->val[(size_t)e] * cv.at((size_t)(cols[b] * n_col + P->col[(size_t)e]));
                    }
                    for (size_t a = 0; a < rows.size(); ++a) {
                        const size_t ia = side ? b : a, ib = side ? a : b;
                        ev.at((size_t)g.eval0 + ia * g.mn.size() + ib) +=
                            y * rv.at((size_t)(rows[a] * n_row + P->row_id[(size_t)r]));
                    }
                }
            }
    double worst = 0;
    for (int c = 0; c < L.n_comp; ++c) {
        cd v = 0;
        for (int e = P->comp_off[(size_t)c]; e < P->comp_off[(size_t)c + 1]; ++e) v += ev.at((size_t)P->comp_eval[(size_t)e]);
        v *= P->scale * L.parts[0].norm;  // the chain's sums are not normalised
        const double scale = mag[(size_t)c] > 0 ? mag[(size_t)c] : 1.0;
        worst = std::max(worst, std::abs(v - C[(size_t)c]) / scale);
    }
    std::printf("%s: pair form, %zu groups, %zu entries, %zu x %d products, worst difference %.1e\n", name,
                P->groups.size(), P->col.size(), P->masks2.size(), P->n_rows2, worst);
    return worst > 1e-10;
}

// every output of a pn step equals the one that stands for its mirror pair
static int bad_mirror(const char *name, const mbc_term_list &L, bool expect, std::mt19937 &rng) {
    const auto P = mbc::mirror_plan(&L);
    if (!!P != expect) {
        std::printf("%s: mirror pairs %s\n", name, P ? "made" : "not made");
        return 1;
    }
    if (!P) return 0;
    std::normal_distribution<double> nd;
    std::vector<cd> f((size_t)L.block_size), z;
    for (auto &v : f) v = cd(nd(rng), nd(rng));
    const auto &s = L.steps[0];
    for (int64_t i = 0; i < s.n_z; ++i) {
        cd v = 0;
        for (int64_t j = i * s.k; j < (i + 1) * s.k; ++j) {
            const cd t = f[s.x[(size_t)j]] * f[s.ys[(size_t)j] & 0x7fff];
            v += s.ys[(size_t)j] & 0x8000 ? -t : t;
        }
        z.push_back(v);
    }
    double worst = 0;
    for (int64_t i = 0; i < s.n_z; ++i)
        worst = std::max(worst, std::abs(z[(size_t)i] - z[(size_t)P->keep.at((size_t)P->rep.at((size_t)i))]));
    std::printf("%s: %zu of %lld outputs, worst difference %.1e\n", name, P->keep.size(), (long long)s.n_z, worst);
    return worst > 1e-11;
}

static mbc_op_spec spec(int np, int nn, int D) {
    mbc_op_spec s;
    std::memset(&s, 0, sizeof(s));
    s.n_p = np;
    s.n_n = nn;
    s.dirac_dim = D;
    s.n_sources = s.n_sinks = 1;
    return s;
}

int main() {
    std::mt19937 rng(7);
    int bad = 0;
    auto build1 = [](const mbc_op_spec &s) {
        mbc_term_list *L = nullptr;
        mbc_build_term_list(&s, &L);
        return L;
    };
    struct Case {
        const char *name;
        int np, nn, D, list_free;
        bool minors;
    };
    for (const Case &c : {Case{"3He", 2, 1, 2, 0, true}, Case{"3H", 1, 2, 2, 0, true}, Case{"4He", 2, 2, 2, 0, true},
                          Case{"pn", 1, 1, 2, 0, false}, Case{"pn rel", 1, 1, 4, 0, false}}) {
        mbc_op_spec s = spec(c.np, c.nn, c.D);
        s.list_free = c.list_free;
        mbc_term_list *L = build1(s);
        bad += bad_minors(c.name, *L, c.minors, rng);
        bad += bad_pairs(c.name, *L, true, rng);
        bad += bad_mirror(c.name, *L, c.np == 1 && c.nn == 1, rng);
        mbc_free_term_list(L);
    }
    for (int o = 0; o < 2; ++o) {  // listed components, both paths
        const int8_t snk[6] = {0, 1, 1, 1, 1, 0}, src[6] = {0, 0, 1, 0, 0, 1}, path[2][2] = {{0, 1}, {1, 0}};
        mbc_op_spec s = spec(1, 1, 2);
        s.spin_mode = MBC_SPIN_LISTED;
        s.n_spin_sel = 3;
        s.snk_spins = snk;
        s.src_spins = src;
        s.path = path[o];
        s.path_len = 2;
        mbc_term_list *L = build1(s);
        bad += bad_mirror("pn listed", *L, true, rng);
        mbc_free_term_list(L);
    }
    {  // pair forms: listed components, odd spin orders, sinks and sources, paths
        struct Listed {
            const char *name;
            int np, nn, D, ns, nk, n;
            std::vector<int8_t> snk, src;
            std::vector<int8_t> path;
        };
        for (const Listed &c : {
                 Listed{"4He rel", 2, 2, 4, 1, 1, 1, {0, 1, 0, 1}, {0, 1, 0, 1}, {}},
                 Listed{"4He rel, two listed", 2, 2, 4, 1, 1, 2, {0, 1, 0, 1, 2, 0, 1, 3}, {0, 1, 0, 1, 0, 1, 0, 1}, {}},
                 Listed{"4He rel, exchanged", 2, 2, 4, 1, 1, 2, {0, 1, 0, 2, 0, 2, 0, 1}, {0, 1, 1, 3, 1, 3, 0, 1}, {0, 1, 0, 1}},
                 Listed{"3He rel", 2, 1, 4, 1, 1, 2, {0, 1, 2, 0, 3, 1}, {0, 1, 0, 0, 1, 2}, {}},
                 Listed{"3H rel", 1, 2, 4, 1, 1, 1, {2, 0, 1}, {0, 0, 1}, {1, 0, 1}},
                 Listed{"4He two sources, two sinks", 2, 2, 2, 2, 2, 2, {0, 1, 2, 3, 0, 2, 0, 2}, {0, 2, 0, 2, 0, 2, 0, 2}, {}},
                 Listed{"3He two sources", 2, 1, 2, 2, 1, 2, {0, 1, 0, 0, 1, 1}, {0, 1, 2, 1, 3, 0}, {}}}) {
            mbc_op_spec s = spec(c.np, c.nn, c.D);
            s.n_sources = c.ns;
            s.n_sinks = c.nk;
            s.spin_mode = MBC_SPIN_LISTED;
            s.n_spin_sel = c.n;
            s.snk_spins = c.snk.data();
            s.src_spins = c.src.data();
            s.path = c.path.empty() ? nullptr : c.path.data();
            s.path_len = (int)c.path.size();
            mbc_term_list *L = build1(s);
            bad += bad_pairs(c.name, *L, true, rng);
            mbc_free_term_list(L);
        }
        mbc_op_spec s = spec(2, 0, 4);  // one species alone
        mbc_term_list *L = build1(s);
        bad += bad_pairs("pp", *L, false, rng);
        mbc_free_term_list(L);
        s = spec(2, 2, 2);
        s.list_free = 1;
        L = build1(s);
        bad += bad_pairs("4He list-free", *L, false, rng);
        mbc_free_term_list(L);
    }
    {  // a projection: several sink and source sets with weights in one output
        const int8_t snk[9] = {1, 0, 0, 0, 1, 1, 0, 1, 0}, src[9] = {0, 1, 0, 0, 1, 1, 1, 0, 1};
        const int32_t to[3] = {0, 0, 1};
        const double w[3] = {0.5, -0.25, 1.5};
        mbc_op_spec s = spec(2, 1, 2);
        s.spin_mode = MBC_SPIN_PROJECTED;
        s.n_spin_sel = 3;
        s.n_proj = 2;
        s.snk_spins = snk;
        s.src_spins = src;
        s.term_proj = to;
        s.term_coef = w;
        mbc_term_list *L = build1(s);
        bad += bad_minors("3He projections", *L, true, rng);
        bad += bad_pairs("3He projections", *L, true, rng);
        mbc_free_term_list(L);
    }
    {  // a projection over every source set: rows of up to 1,311 entries
        std::vector<int8_t> snk, src;
        std::vector<int32_t> to;
        std::vector<double> w;
        for (int8_t a = 0; a < 4; ++a)
            for (int8_t b = (int8_t)(a + 1); b < 4; ++b)
                for (int8_t c = 0; c < 4; ++c) {
                    for (int8_t v : {0, 1, 0}) snk.push_back(v);
                    for (int8_t v : {a, b, c}) src.push_back(v);
                    to.push_back(0);
                    w.push_back(0.25 + 0.125 * (double)to.size());
                }
        mbc_op_spec s = spec(2, 1, 4);
        s.spin_mode = MBC_SPIN_PROJECTED;
        s.n_spin_sel = (int)to.size();
        s.n_proj = 1;
        s.snk_spins = snk.data();
        s.src_spins = src.data();
        s.term_proj = to.data();
        s.term_coef = w.data();
        mbc_term_list *L = build1(s);
        bad += bad_pairs("3He rel, every source set", *L, true, rng);
        mbc_free_term_list(L);
    }
    {  // two nuclei on one path, both orders of adding baryons
        for (int o = 0; o < 2; ++o) {
            const int8_t path[2][4] = {{0, 0, 1, 1}, {0, 1, 0, 1}};
            mbc_op_spec s[2] = {spec(2, 1, 2), spec(2, 2, 2)};
            s[1].path = path[o];
            s[1].path_len = 4;
            mbc_term_list *L = nullptr;
            mbc_build_combined(s, 2, &L);
            bad += bad_minors("3He and 4He on one path", *L, true, rng);
            mbc_free_term_list(L);
        }
    }
    {  // 8Be: L^2 = 1,814,400^2; an odd order of the sink spins flips the sign
        const int8_t snk[16] = {0, 1, 2, 3, 0, 1, 2, 3, 1, 0, 2, 3, 0, 1, 2, 3};
        const int8_t src[16] = {0, 1, 2, 3, 0, 1, 2, 3, 0, 1, 2, 3, 0, 1, 2, 3};
        mbc_op_spec s = spec(4, 4, 4);
        s.spin_mode = MBC_SPIN_LISTED;
        s.n_spin_sel = 2;
        s.snk_spins = snk;
        s.src_spins = src;
        s.list_free = 1;
        mbc_term_list *L = build1(s);
        const auto P = mbc::saturated_plan(L);
        const double K = 1814400.0 * 1814400.0;
        const bool ok = P && P->coef.size() == 2 && P->coef[0] == K && P->coef[1] == -K;
        std::printf("8Be: saturated form %s\n", ok ? "as expected" : "wrong");
        bad += !ok;
        mbc_free_term_list(L);
        L = build1(spec(2, 2, 2));
        bad += mbc::saturated_plan(L) != nullptr;
        mbc_free_term_list(L);
    }
    std::printf("%s\n", bad ? "FAIL" : "OK");
    return bad ? 1 : 0;
}

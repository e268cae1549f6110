// Host check of lists read from files: an unchanged file gets the plans of the list
// that was written; one whose operations are not the recursion's gets none, so its
// own operations are evaluated. argv[1]: a scratch file.
#include <cstdio>
#include <functional>

#include "../../paper_1301_4895_gb300/csrc/builder.cpp"
#include "../../paper_1301_4895_gb300/csrc/list_io.cpp"
#include "../../paper_1301_4895_gb300/csrc/plan.cpp"

namespace mbc {
void free_device_cache(mbc_term_list *) {}
}  // namespace mbc

struct Spec : mbc_op_spec {
    Spec(int np, int nn, int D) : mbc_op_spec{} {
        n_p = np;
        n_n = nn;
        dirac_dim = D;
        n_sources = n_sinks = 1;
    }
};

// bits of the plans that a list gets
static int plans(const mbc_term_list *L) {
    return (mbc::minor_plan(L) ? 1 : 0) | (mbc::pair_plan(L) ? 2 : 0) | (mbc::mirror_plan(L) ? 4 : 0) |
           (mbc::saturated_plan(L) ? 8 : 0);
}

int main(int, char **argv) {
    using Edit = std::function<void(mbc_term_list &)>;
    const int8_t he4[4] = {0, 1, 0, 1}, be8[8] = {0, 1, 2, 3, 0, 1, 2, 3};
    Spec rel(2, 2, 4), sat(4, 4, 4);
    rel.spin_mode = sat.spin_mode = MBC_SPIN_LISTED;
    rel.n_spin_sel = sat.n_spin_sel = 1;
    rel.snk_spins = rel.src_spins = he4;
    sat.snk_spins = sat.src_spins = be8;
    sat.list_free = 1;
    const struct {
        const char *name;
        Spec spec;
    } lists[] = {{"3He", Spec(2, 1, 2)}, {"pn", Spec(1, 1, 2)}, {"4He rel", rel}, {"8Be list-free", sat}};
    const struct {
        const char *name;
        bool stored;  // an edit of stored operations
        Edit edit;
    } edits[] = {
        {"sign of a later operation", true, [](mbc_term_list &L) { L.steps.back().ys[1] ^= 0x8000; }},
        {"an operation twice", true,
         [](mbc_term_list &L) {
             mbc::Step &s = L.steps.back();
             s.x[1] = s.x[0];
             s.ys[1] = s.ys[0];
         }},
        {"another input", true,
         [](mbc_term_list &L) {
             mbc::Step &s = L.steps[0];
             s.x[(size_t)s.k] = (uint32_t)((s.x[(size_t)s.k] + 1) % (uint32_t)s.n_x);
         }},
        {"set sizes of a generated step", false, [](mbc_term_list &L) { std::swap(L.steps[3].xk[0], L.steps[3].xk[1]); }},
    };
    int bad = 0;
    for (const auto &l : lists) {
        mbc_term_list *L = nullptr, *back = nullptr;
        if (mbc_build_term_list(&l.spec, &L) != MBC_OK || mbc_save_term_list(L, argv[1]) != MBC_OK) return 1;
        const int want = plans(L);
        mbc_free_term_list(L);
        if (mbc_load_term_list(argv[1], &back) != MBC_OK) return 1;
        const int got = plans(back);
        std::printf("%s: plans %d, from the file %d\n", l.name, want, got);
        bad += !want || got != want;
        mbc_free_term_list(back);
        for (const auto &e : edits) {
            if (e.stored == (l.spec.list_free != 0)) continue;
            if (mbc_load_term_list(argv[1], &back) != MBC_OK) return 1;
            e.edit(*back);
            const int p = plans(back);
            std::printf("%s, %s: plans %d\n", l.name, e.name, p);
            bad += p != 0;
            mbc_free_term_list(back);
        }
    }
    std::printf("%s\n", bad ? "FAIL" : "OK");
    return bad ? 1 : 0;
}

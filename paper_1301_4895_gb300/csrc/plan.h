// Evaluation plans derived from a built term list (host only). A list fixes
// which components it yields and the source tensor L of each; these plans are
// cheaper formulas for the same components than the list's own operations,
// used where the sink is a point. Not part of the public ABI.
#pragma once

#include <cstdint>
#include <memory>
#include <vector>

#include "mbc_internal.h"

namespace mbc {

// A component key: proton spins, neutron spins, u and d quark index sets.
struct PlanKey {
    uint32_t dp, dn, u, d;
};

// One nonzero entry of a component's contraction list with its key.
struct PlanEntry {
    PlanKey z;
    double l;
};

// Contraction entries of every component with their keys, read back from the
// first operation (or the rank) of each output. False where those do not have the
// component's numbers of quarks and baryons, or an L value is not finite.
bool list_entries(const mbc_term_list &L, std::vector<std::vector<PlanEntry>> &comp);

// True where every output of the list has all splits of its key, each once and
// with its sign, so that a formula of the keys gives what the operations give.
// A file can hold any operations that stay in bounds; the builder's are complete.
// List-free steps with index tables are not looked through: false. 8Be's stored
// operations (448 M) take 0.9 s on 8 cores, 4He's with one component 20 ms.
bool complete_operations(const mbc_term_list &L);

// The sink (or unit-propagator) tensor of k baryons of one species with the
// given spin set: nonzero values of the ordered product of the G tensors as
// (pair-flavour mask, single-flavour mask, value). For protons the pair
// flavour is u; the neutron tensor holds the same numbers with u and d
// exchanged, since Gamma_2 and epsilon are both antisymmetric.
struct SpeciesEntry {
    uint32_t pair, single;
    int64_t v;
};
std::vector<SpeciesEntry> species_tensor(int dim, uint32_t spins);

// Minor form of a point-sink list: a component's quark sets factorise into
// flavours, F[sigma; U, D] = sum L_sink(sigma; U', D') det S[U', U] det S[D', D],
// so a correlator is a weighted sum of products of two minors of the site's
// propagator tile (the same tile for both flavours). Minors are built order by
// order by Laplace expansion, only those some term needs.
//   region 1 is the tile itself (entry row * nxi + column); region o holds the
//   needed minors of order o. steps[i] builds region z from products of
//   entries of regions x and y, k per output, z-major.
//   Component c is the sum over its runs [run_off[c], run_off[c+1]) of
//   run_coef * sum of +- products, terms [term_off[r], term_off[r+1]).
struct MinorPlan {
    struct Step {
        int x_reg, y_reg, z_reg;
        int32_t n_z, k;
        std::vector<uint16_t> x, y;
        std::vector<uint8_t> neg;
    };
    struct Term {
        uint8_t x_reg, y_reg;
        uint16_t x, y;
        bool neg;
    };
    int32_t reg_size[8] = {0};
    std::vector<Step> steps;
    std::vector<int32_t> run_off, term_off;
    std::vector<double> run_coef;
    std::vector<Term> terms;
};

// The minor plan of a list, made once per list; nullptr where the list does
// not qualify (several sources or sink functions, relativistic operators; more
// than kMaxMinorRuns runs or kMaxMinorRows minors of an order) or where its own
// operations are fewer, its block included: 3He takes 1,860 complex multiply-adds
// per site as minors against 7,560, 4He 187 against 12,492, while pn's 6,784 exceed
// its recursion's 4,176. Measured on GB300, 3He and 4He on 16^3 x 32 sites: FP64
// 18.42 -> 2.12 ms, mixed 2.05 -> 0.46 ms.
std::shared_ptr<const MinorPlan> minor_plan(const mbc_term_list *L);

// Saturated form of a relativistic point-sink list: where every contracted
// component takes all 12 u and all 12 d indices (8Be), the only minors left are
// the determinants, C_c = coef[c] det S_u det S_d (Sec. 8), coef[c] the
// contraction of the two tensors' single entries.
struct SaturatedPlan {
    std::vector<double> coef;
};
std::shared_ptr<const SaturatedPlan> saturated_plan(const mbc_term_list *L);

// Pair form of a nucleus with one or two baryons of each species. The protons'
// product P[sigma; a, e] (a: u set, e: d set) and the neutrons' N (the same
// numbers for u = d, with the flavours exchanged) are formed once per spin set,
// ordered (f_{s1} ^ f_{s2}, s1 < s2: the recursion adds both orders, which are
// equal), and a component is bilinear in them,
//   C = sum_z L(z) F(z) = sum_{i, j} P_i Lambda_ij N_j,
// Lambda_ij = +-L(a_i + g_j, b_j + e_i) real, sparse and the same for every
// site. Components with the same L share a group. Exchanging the flavours maps
// (sigma_p, sigma_n, L(U, D)) to (sigma_n, sigma_p, L(D, U)) with the same
// value, so only one of the two is computed, and a symmetric Lambda keeps each
// pair (i, j) once, <P_a, T P_b> + <P_b, T P_a>.
//   Every entry belongs to a row: a P row i that gathers N_b[j] (y_b = sum_j
// Lambda_ij N_b[j], then P_a[i] y_b for every proton set a), or an N row j that
// gathers P_a[i]. A row costs sets_p x sets_n products however few entries it
// has, so a greedy vertex cover picks the rows (half of them in 4He with all
// components). Lambda splits into about a thousand blocks of at most 285 rows
// that share no column; rows are ordered by colour content (28 classes, which a
// row's entries share), block and columns, so that the rows of neighbouring
// warps gather the same entries.
// Gathered entries that a pack of rows names at most (k_pair): with two spin sets
// 204 rows of 512 B fill an SM's shared memory; one set takes half of it, so two
// CTAs overlap one's copies with the other's sums. No row is longer (88 entries in
// 4He with all components; projections over many source sets reach 1,311, in pieces).
constexpr int kPackCols = 204;
struct PairPlan {
    int np = 0, nn = 0;  // baryons per species: 1 or 2
    // two-baryon products: element m (spin set masks2[m]), row r at m * n_rows2 +
    // r. Rows with the same two singles (e0, e1) are consecutive: range k is
    // rows [range_off[k], range_off[k + 1]) with singles range_e[k] = e0 | e1 << 8.
    // A row of quark set {a, b, c, d} is the sum over its splits into two pairs and
    // both orders of the singles of a lower-spin block f times an upper-spin block
    // g, the same for every spin set: 12 products. Rows of a range that share a
    // triple {a, b, c} form runs (ProdRun): the pairs within the triple are operands
    // of all of them. Range k has runs [run_off[k], run_off[k + 1]); a run's rows are
    // prod_rec[rec0 .. rec0 + n): cd | bd << 7 | ad << 14 (the pairs opposite to
    // ab, ac and bc) | row within the range << 21 | odd split << 30, the one of the
    // three splits whose sign is negative.
    static constexpr int kProdRun = 9;  // rows of a run at most: the other quark states
    struct ProdRun {
        uint32_t rec0;
        uint8_t n, pair[3];  // ab, ac, bc
    };
    std::vector<uint32_t> masks2;
    int32_t n_rows2 = 0;
    std::vector<ProdRun> prod_runs;
    std::vector<uint32_t> prod_rec;
    std::vector<int32_t> run_off;
    std::vector<int32_t> range_off;
    std::vector<uint16_t> range_e;
    struct Group {
        int64_t row0[2], row1[2];       // its rows in row_id / row_ptr: P rows, N rows
        std::vector<int32_t> mp, mn;    // element indices; every (mp, mn) is evaluated
        int64_t eval0;                  // evaluation (mp_i, mn_j) at eval0 + i * mn.size() + j
    };
    std::vector<Group> groups;
    std::vector<uint32_t> row_id;       // P (or N) row of each Lambda row
    std::vector<uint16_t> row_class;    // colour content of the row
    std::vector<int64_t> row_ptr;       // its entries (one more than row_id)
    std::vector<uint32_t> col;          // N (or P) row of each entry
    std::vector<double> val;
    bool val_fp32 = true;               // every value is an FP32 number
    int64_t n_evals = 0;
    std::vector<int32_t> comp_off;      // evaluations a component sums (n_comp + 1)
    std::vector<int32_t> comp_eval;
    double scale = 1.0;                 // n_P! n_N! / norm
    int64_t p_rows(int64_t block_rows) const { return np == 2 ? n_rows2 : block_rows; }
    int64_t n_rows(int64_t block_rows) const { return nn == 2 ? n_rows2 : block_rows; }
};
std::shared_ptr<const PairPlan> pair_plan(const mbc_term_list *L);

// Mirror pairs of a pn list's outputs: exchanging the flavours maps the component
// (sigma_p, sigma_n; U, D) to (sigma_n, sigma_p; D, U) of the same value (u = d),
// so the step keeps one of each pair: 154 of 296 outputs for the nonrelativistic
// list with all components (pn, 4^3 x 8: 41.0 -> 30.8 us).
struct MirrorPlan {
    std::vector<int32_t> keep;  // outputs computed
    std::vector<int32_t> rep;   // per output, position in keep
};
std::shared_ptr<const MirrorPlan> mirror_plan(const mbc_term_list *L);

}  // namespace mbc

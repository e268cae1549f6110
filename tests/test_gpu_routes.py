"""GPU parity at the edges of the contraction's routes: tile remainders, the site
counts where a launch rule changes kernel, and the forms (minors, determinant,
pair products, line sums) on shapes where they can go wrong. Bounds as in
test_gpu_parity (parity.check); closed forms as its full-slab test."""
import numpy as np
import pytest

import parity
import synth
from gpu_helpers import EPS, legs, oracle_plan, oracle_slab
from parity import TOL
from test_gpu_parity import (BE8, _be8_K, _check_sparse, check_legs, mbc, run,  # noqa: F401  (mbc is the fixture)
                             test_spin_projection_outputs as check_projections)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 3, 5), (14, 14, 13)])
def test_saturated_few_and_many_sites(mbc, dims):
    """8Be by one determinant per site, four warps per site (few sites) and half a
    warp (more than 16 per SM: 2,548 sites), three momenta."""
    from oracle import site_sum
    field = synth.field(40, 1, 2, dims, 0.1, eps=0.02)
    tl = mbc.build_term_list(4, 4, 4, spins=[(BE8, BE8)], list_free=True)
    moms = ((0, 0, 0), (1, 0, 0), (0, 2, 1))
    for p in (0, 1):
        got = run(mbc, field, [tl], p, moms=moms)
        for t in range(2):
            C = _be8_K() * np.linalg.det(field[0, t].reshape(-1, 12, 12)) ** 2
            ref = site_sum.site_sum(C[:, None], synth.site_coords(dims), tuple(dims[::-1]), list(moms))[:, 0]
            # sum|terms| <= 10 |C| at eps = 0.02, as in the full-slab test
            assert np.max(np.abs(got[0, 0, t, :, 0] - ref)) <= 10 * TOL[p] * np.sum(np.abs(C)), (p, t)


@pytest.mark.parametrize("dims", [(1, 2, 3), (14, 14, 13)])
def test_saturated_pivoting_and_singular_sites(mbc, dims):
    """Row permutations (every pivot off the diagonal), a zero row, a zero matrix
    and entries whose squares leave the exponent range."""
    n = int(np.prod(dims))
    rng = np.random.default_rng(41)
    S = np.zeros((n, 12, 12), dtype=np.complex128)
    perm = rng.permutation(12)
    S[0] = np.eye(12)[perm] * 1.5
    S[1] = rng.standard_normal((12, 12)) + 1j * rng.standard_normal((12, 12))
    S[1, 7] = 0
    S[2] = np.diag([1e-200, 1e200] + [1.0] * 10)
    S[n - 1] = np.eye(12)[perm[::-1]] * 1j
    tl = mbc.build_term_list(4, 4, 4, spins=[(BE8, BE8)], list_free=True)
    ref = _be8_K() * (1.5 ** 24 + 0.0 + 1.0 + 1.0)  # det^2: 1.5^24, 0, 1, i^24
    for p in (0, 1):
        got = run(mbc, S.reshape((1, 1) + dims + (12, 12)), [tl], p)[0, 0, 0, 0, 0]
        if p == 0:
            assert abs(got - ref) <= 1e-12 * abs(ref)
        assert np.isfinite(got.real)


@pytest.mark.parametrize("dims", [(1, 1, 31), (3, 11, 1), (1, 5, 13)])
def test_minor_form_tile_remainders(mbc, dims):
    """31, 33 and 65 sites: 3He, 3H and 4He around the 32-site tiles."""
    lists = [mbc.build_term_list(2, 1, 2), mbc.build_term_list(1, 2, 2), mbc.build_term_list(2, 2, 2)]
    check_legs(mbc, 42, 1, 1, dims, 0.3, lists, [(2, 1, 2), (1, 2, 2), (2, 2, 2)], moms=((0, 0, 0), (1, 0, 2)))


@pytest.mark.parametrize("n_p,n_n", [(2, 1), (2, 2), (1, 1)])
def test_small_kernels_on_more_tiles_than_sms(mbc, n_p, n_n):
    """17^3 sites (a ragged last tile, more tiles than SMs): FP64 minors with lanes
    as sites, the tile sums of several warps."""
    _check_sparse(mbc, 43, (17, 17, 17), 0.4, [0, 31, 32, 2500, 4912], mbc.build_term_list(n_p, n_n, 2), (n_p, n_n, 2))


@pytest.mark.parametrize("n_p,n_n,spins", [
    (1, 1, None),
    (2, 1, [((0, 1, 2), (0, 1, 0)), ((0, 3, 1), (0, 1, 2))]),
    (1, 2, [((2, 0, 1), (0, 0, 1))]),
    (2, 2, [((0, 1, 0, 1), (0, 1, 0, 1)), ((0, 1, 0, 2), (0, 1, 0, 1))]),
    (2, 2, [((0, 1, 0, 2), (0, 1, 1, 3)), ((0, 2, 0, 1), (1, 3, 0, 1)), ((2, 3, 0, 1), (0, 1, 1, 3))]),
])
def test_pair_form_relativistic(mbc, n_p, n_n, spins):
    """Pair form with one and two baryons per species, one to six spin sets per
    tile, exchanged flavours and a symmetric matrix; 65 sites (a tile and one)."""
    dims = (1, 5, 13)
    tl = mbc.build_term_list(n_p, n_n, 4, spins=spins)
    check_legs(mbc, 44, 1, 1, dims, 0.3, [tl], [(n_p, n_n, 4)], moms=((0, 0, 0), (0, 1, 2)))


def test_pair_form_long_rows(mbc):
    """A projection over every source set: Lambda rows of up to 1,311 entries, more
    than a pack of gathered rows holds (the weights exact in FP32)."""
    sources = [(a, b, c) for a in range(4) for b in range(a + 1, 4) for c in range(4)]
    terms = [((0, 1, 0), src, 0.25 + 0.125 * k) for k, src in enumerate(sources)]
    check_projections(mbc, 2, 1, 4, [terms])


@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 2, 7), (2, 5, 3)])
@pytest.mark.parametrize("n_p,n_n,D,spins", [(2, 1, 2, None), (1, 1, 4, [((0, 3), (1, 2)), ((2, 2), (0, 1))])])
def test_projection_lines_and_passes(mbc, dims, n_p, n_n, D, spins):
    """Line sums on odd extents with 7 momenta: two passes, up to four distinct n_x
    in one, some equal modulo the extent."""
    from oracle import projection
    moms = ((0, 0, 0), (1, 0, 0), (2, 1, 0), (-1, 0, 3), (7, 1, 1), (0, 2, 1), (1, 1, 1))
    tl = mbc.build_term_list(n_p, n_n, D, spins=spins)
    comps = tl.components()
    plan = oracle_plan(n_p, n_n, D, comps)
    for field, precs in legs(45, 1, 2, dims, 0.3, gauss=False):
        for p in precs:
            got = run(mbc, field, [tl], p, moms=moms, sink=mbc.SINK_BLOCK_MOMENTUM)
            for t in range(2):
                C, sc = projection.projected_correlators(plan, field[0, t], dims, moms)
                parity.check(got[0, 0, t, :, : len(comps)], C, sc, p, what=f"lines {dims} ({n_p},{n_n}) t {t}")


@pytest.mark.parametrize("spins", [
    [((0, 1, 0, 2), (0, 1, 1, 3)), ((0, 2, 0, 1), (1, 3, 0, 1)), ((2, 3, 0, 1), (0, 1, 1, 3))],
    [((0, 1, 0, 2), s) for s in ((0, 1, 0, 1), (0, 1, 0, 2), (0, 2, 0, 3), (0, 3, 1, 2), (1, 2, 1, 3))],
])
def test_projected_items_around_the_fp64_rule(mbc, spins):
    """Mixed projected blocks whose pair form has 1.7 M and 2.3 M multiply-adds an
    item: contracted in FP64 and in FP32."""
    from oracle import projection
    dims, moms = (1, 2, 3), ((0, 0, 0), (1, 1, 0))
    tl = mbc.build_term_list(2, 2, 4, spins=spins)
    assert (tl.form(mbc.SINK_BLOCK_MOMENTUM, 1)[1] <= 8 * 2e6) == (len(spins) == 3)
    comps = tl.components()
    plan = oracle_plan(2, 2, 4, comps)
    for field, precs in legs(48, 1, 1, dims, 0.3, gauss=False):
        C, sc = projection.projected_correlators(plan, field[0, 0], dims, moms)
        for p in precs:
            got = run(mbc, field, [tl], p, moms=moms, sink=mbc.SINK_BLOCK_MOMENTUM)[0, 0, 0, :, : len(comps)]
            parity.check(got, C, sc, p, what=f"projected items, {len(spins)} components")


def test_zero_momentum_without_phase_table(mbc):
    """Calls at zero momentum alone use no phase table: the same bits as the zero
    momentum of a call with others."""
    dims = (3, 5, 7)
    field = synth.field(46, 1, 2, dims, 0.3, eps=EPS)
    sp = (0, 1, 0, 1)
    lists = [mbc.build_term_list(1, 1, 2), mbc.build_term_list(2, 1, 2), mbc.build_term_list(2, 2, 4, spins=[(sp, sp)])]
    for p in (0, 1):
        one = run(mbc, field, lists, p)
        two = run(mbc, field, lists, p, moms=((0, 0, 0), (1, 0, 2)))
        assert np.array_equal(one[..., 0, :], two[..., 0, :]), p


def test_pair_form_captured_after_a_forced_recursion(mbc):
    """A list's first call uploads what its other calls read: the default form is
    captured after a warm call that forced the recursion (scratch grown by another
    list of the same sizes)."""
    import torch
    dims, sp = (1, 5, 13), (0, 1, 0, 1)
    field = torch.from_numpy(synth.field(47, 1, 1, dims, 0.3, eps=EPS)).cuda()
    a, b = (mbc.build_term_list(2, 2, 4, spins=[(sp, sp)]) for _ in range(2))
    st = torch.cuda.Stream()
    out = torch.zeros((1, 1, 1, 1, 1), dtype=torch.complex128, device="cuda")
    mbc.contract(field, [a], stream=st, out=out)
    mbc.contract(field, [b], stream=st, out=out, tune={"regime": 2})
    st.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        mbc.contract(field, [b], stream=st, out=out)
    out.zero_()
    g.replay()
    ref = mbc.contract(field, [a], stream=st)
    torch.cuda.synchronize()  # ref is made on st, compared on the current stream
    assert torch.equal(out, ref)


def test_block_slices_on_two_relativistic_sources(mbc):
    """24-column tiles (triangular diquarks, entry slices) on pn, 5 sites."""
    from oracle import gamma, recursion
    dims = (1, 1, 5)
    spins = [((0, 3), (1, 6)), ((2, 1), (0, 3))]
    tl = mbc.build_term_list(1, 1, 4, spins=spins, n_sources=2)
    comps = tl.components()
    plan = recursion.Plan(1, 1, 4, requests=comps, G=gamma.g_tensor_sources(4, 2), G_sink=gamma.g_tensor(4))
    for field, precs in legs(47, 1, 1, dims, 0.3, n_src=2):
        ref, scale = oracle_slab(plan, recursion.source_columns(field[0, 0], 4), dims, [(0, 0, 0)])
        for p in precs:
            got = run(mbc, field, [tl], p)[0, 0, 0, :, : len(comps)]
            parity.check(got, ref, scale[None, :], p, what="24 columns")


@pytest.mark.parametrize("build,dims,nt,precs", [
    # 8Be: 1,728 sites a slab by four warps a site, 5,184 by half a warp
    (lambda m: [m.build_term_list(4, 4, 4, spins=[(BE8, BE8)], list_free=True)], (12, 12, 12), 3, (0, 1)),
    # clusters of four CTAs: 3 sites a slab
    (lambda m: [m.build_term_list(4, 4, 4, spins=[(BE8, BE8)], list_free=True)], (1, 1, 3), 4, (0, 1)),
    # nonrelativistic lists in mixed precision: 64 tiles of 32 sites, 64 outputs a slab
    (lambda m: [m.build_term_list(1, 1, 2), m.build_term_list(2, 1, 2), m.build_term_list(2, 2, 2)], (16, 16, 8), 6, (1,)),
    # pair form: waves of 64 and of 1,024 sites; 18 tiles and 256 outputs a slab
    (lambda m: [m.build_term_list(2, 2, 4, spins=[((0, 1, 0, 1), (0, 1, a, b)) for a in range(4) for b in range(a)])],
     (4, 4, 4), 16, (0, 1)),
    (lambda m: [m.build_term_list(1, 1, 4)], (9, 8, 8), 2, (1,)),
])
def test_a_slab_alone_and_among_others(mbc, build, dims, nt, precs):
    """A slab's correlators have the same bits whether the call holds that slab alone,
    as a rank of a sharded run may, or all of them."""
    moms = ((0, 0, 0), (1, 0, 0), (0, 1, 0), (1, 1, 0))
    field, lists = synth.field(49, 1, nt, dims, 0.1, eps=EPS), build(mbc)
    for p in precs:
        whole = run(mbc, field, lists, p, moms=moms)
        for t in range(nt):
            alone = run(mbc, field, lists, p, moms=moms, t0=t, t1=t + 1)
            assert np.array_equal(alone[:, :, 0], whole[:, :, t]), (p, t)


def test_mixed_projection_across_the_lines(mbc):
    """Mixed projected blocks at a momentum across the lattice lines: a line's sum and
    its phase keep both words. Median error against FP64 over 256 slabs; rounded to one
    word it is 1.6e-6 (on 7 lines the phases' roundings do not cancel), else 0.7e-6."""
    sp = (0, 1, 0, 1)
    tl = mbc.build_term_list(2, 2, 4, spins=[(sp, sp)])
    field = synth.field(50, 2, 128, (5, 7, 9), 0.0, eps=EPS)
    exact, got = (run(mbc, field, [tl], p, moms=((0, 1, 0),), sink=mbc.SINK_BLOCK_MOMENTUM) for p in (0, 1))
    assert np.median(np.abs(got - exact) / np.abs(exact)) <= 1.0e-6


def test_be8_recursion_on_request(mbc):
    """8Be by its recursion: stored operations, the same regenerated on request (which
    default tuning honours too), and a list-free list. On near-identity propagators,
    against O3; the three perform the same operations."""
    dims = (1, 2, 2)
    field = synth.field(4, 1, 1, dims, 0.4, dtype=np.complex64, eps=EPS)
    stored, free = (mbc.build_term_list(4, 4, 4, spins=[(BE8, BE8)], list_free=lf) for lf in (False, True))
    ref, scale = oracle_slab(oracle_plan(4, 4, 4, [(BE8, BE8)]), field[0, 0], dims, [(0, 0, 0)])
    for p in (0, 1):
        a = run(mbc, field, [stored], p, tune={"regime": 2})
        parity.check(a[0, 0, 0, :, :1], ref, scale[None, :], p, what="8Be recursion")
        for tl, tune in ((stored, {"regime": 2, "list_free": 1}), (stored, {"list_free": 1}), (free, {"regime": 2})):
            b = run(mbc, field, [tl], p, tune=tune)
            if p == 0:
                assert np.array_equal(a, b), tune
            parity.check(b[0, 0, 0, :, :1], ref, scale[None, :], p, what=f"8Be recursion {tune}")


@pytest.mark.parametrize("p", [0, 1])
@pytest.mark.parametrize("dims", [(1, 2, 3), (14, 14, 13)])
def test_saturated_form_is_fp64_in_both_precisions(mbc, dims, p):
    """8Be's determinants of a permutation and of a random matrix, a few and many sites."""
    n = int(np.prod(dims))
    rng = np.random.default_rng(51)
    S = np.zeros((n, 12, 12), dtype=np.complex128)
    S[0] = np.eye(12)[rng.permutation(12)] * 1.5
    S[n - 1] = rng.standard_normal((12, 12)) + 1j * rng.standard_normal((12, 12))
    tl = mbc.build_term_list(4, 4, 4, spins=[(BE8, BE8)], list_free=True)
    got = run(mbc, S.reshape((1, 1) + dims + (12, 12)), [tl], p)[0, 0, 0, 0, 0]
    det2 = np.linalg.det(S[[0, n - 1]]) ** 2
    assert abs(got - _be8_K() * np.sum(det2)) <= 1e-12 * _be8_K() * np.sum(np.abs(det2))


def test_autotune_keeps_the_fast_kernel(mbc):
    """FP64 3He + 4He on 16^3 x 12: the library's choice (the minor form with lanes as
    sites) is a fifth faster than every setting of sites_per_cta."""
    import torch
    from paper_1301_4895_gb300.autotune import autotune
    field = torch.from_numpy(synth.field(52, 1, 12, (16, 16, 16), 0.1)).cuda()
    assert autotune(field, [mbc.build_term_list(2, 1, 2), mbc.build_term_list(2, 2, 2)], use_cache=False) == {}


def test_no_room_for_the_pair_tables(mbc):
    """With too little device memory left for a list's pair tables, a call that forces
    the recursion, which does not read them, runs all the same."""
    import torch
    spins = [((0, 1, 0), (a, b, c)) for b in range(4) for a in range(b) for c in range(4)]
    field = torch.from_numpy(synth.field(53, 1, 1, (1, 2, 2), 0.3, eps=EPS)).cuda()
    out = torch.zeros((4, 1, 1, 1, 1, len(spins)), dtype=torch.complex128, device="cuda")
    lists = [mbc.build_term_list(2, 1, 4, spins=spins) for _ in range(4)]

    def call(i):  # bytes of device memory that it took
        before = torch.cuda.mem_get_info()[0]
        mbc.contract(field, [lists[i]], out=out[i], tune={"regime": 2})
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0]

    call(0)  # scratch and kernels
    copy = min(call(1), call(2))  # 8 MB of operations, then 9 MB of pair tables
    filler = torch.empty(((torch.cuda.mem_get_info()[0] - copy + (4 << 20)) >> 21) << 21, dtype=torch.uint8, device="cuda")
    try:
        assert copy - (7 << 20) < torch.cuda.mem_get_info()[0] < copy - (1 << 20)
        call(3)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert torch.equal(out[3], out[0]) and torch.equal(out[1], out[0])


@pytest.mark.parametrize("n_p,n_n,D,spins,sites,bound", [
    (2, 1, 2, None, 4096, 1.00e-7), (2, 2, 2, None, 4096, 1.09e-7), (2, 2, 4, [((0, 1, 0, 1), (0, 1, 0, 1))], 1024, 9.4e-8),
    (2, 2, 4, None, 64, 1.44e-7),
])
def test_mixed_forms_are_no_further_off_than_the_recursion(mbc, n_p, n_n, D, spins, sites, bound):
    """The mixed minor and pair forms against FP64, single near-identity sites: the
    median error stays below that of the mixed recursion on FP32 blocks, which
    contracted with L in FP64 (bound, measured on such sites; the forms 4.8e-8, 9.8e-8,
    6.9e-8 and 9.5e-8)."""
    tl = mbc.build_term_list(n_p, n_n, D, spins=spins)
    field = synth.field(54, 1, sites, (1, 1, 1), 0.0, eps=EPS)
    exact, got = (run(mbc, field, [tl], p) for p in (0, 1))
    err = np.abs(got - exact)[np.abs(exact) > 0] / np.abs(exact)[np.abs(exact) > 0]
    assert np.median(err) <= bound

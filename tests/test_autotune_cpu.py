"""Candidate launch shapes of the autotuner (host logic, no GPU): every
candidate is a valid tuning record, the kernels a list set uses decide which
fields vary, and the item orders are offered per wave step kernel (FP64: 0
and 1; mixed: 0, one CTA of 32 warps per SM on consecutive outputs of one
site group, and 3, 8-warp CTAs with the site groups side by side)."""
import paper_1301_4895_gb300 as mbc
from paper_1301_4895_gb300 import autotune


def _cands(lists, precision):
    return list(autotune.candidates(lists, precision))


def test_candidates_cover_each_regime():
    nonrel = [mbc.build_term_list(2, 1, 2)]
    rel = [mbc.build_term_list(1, 1, 4)]
    for prec in (mbc.FP64, mbc.MIXED):
        for lists in (nonrel, rel, nonrel + rel):
            cands = _cands(lists, prec)
            assert cands and len({tuple(sorted(c.items())) for c in cands}) == len(cands)
            for c in cands:
                assert set(c) <= set(mbc.Tune.FIELDS)
                t = mbc.Tune(**c)  # a record the library takes
                assert all(getattr(t, k) == v and v > 0 for k, v in c.items())
    # nonrelativistic lists only: the shared-memory kernel's shape varies, no wave fields
    assert all(set(c) <= {"sites_per_cta"} for c in _cands(nonrel, mbc.FP64))
    assert all(set(c) <= {"threads_per_cta"} for c in _cands(nonrel, mbc.MIXED))
    # relativistic lists only: wave fields only
    assert all(not ({"sites_per_cta", "threads_per_cta"} & set(c)) for c in _cands(rel, mbc.FP64))


def test_item_orders_per_wave_step_kernel():
    rel = [mbc.build_term_list(1, 1, 4)]
    assert {c.get("wave_order", 0) for c in _cands(rel, mbc.FP64)} == {0, 1}
    assert {c.get("wave_order", 0) for c in _cands(rel, mbc.MIXED)} == {0, 3}


def test_the_librarys_choice_is_a_candidate():
    """FP64 minor-form lists leave their fast kernel where sites_per_cta is set, so the
    candidates hold the library's own choice; in mixed precision the minor form reads
    no field. pn, which runs the recursion there, keeps its shapes."""
    he = [mbc.build_term_list(2, 1, 2), mbc.build_term_list(2, 2, 2)]
    pn, rel = mbc.build_term_list(1, 1, 2), mbc.build_term_list(1, 1, 4)
    for lists in (he, he + [pn], he + [rel]):
        assert {} in _cands(lists, mbc.FP64)
    assert _cands(he, mbc.MIXED) == [{}]
    assert {c["threads_per_cta"] for c in _cands(he + [pn], mbc.MIXED)} == {256, 512, 768, 1024}


def test_cache_key_and_sample_follow_the_form():
    import json

    import numpy as np
    he, rel = [mbc.build_term_list(2, 1, 2)], [mbc.build_term_list(1, 1, 4)]
    field = np.zeros((1, 2, 2, 2, 2, 12, 12), dtype=np.complex128)
    assert json.loads(autotune._key(field, he, mbc.FP64))["forms"] == ["minors"]
    shape = (1, 32, 16, 16, 16, 12, 12)
    assert autotune._slices(shape, he, mbc.FP64, 1, 152) == 10  # 8 x 32 x 152 sites
    assert autotune._slices(shape, he + rel, mbc.FP64, 1, 152) == 2
    assert autotune._slices(shape, he, mbc.MIXED, 1, 152) == autotune._slices(shape, rel, mbc.FP64, 1, 152) == 1
    assert autotune._slices((1, 4) + shape[2:], he, mbc.FP64, 1, 152) == 4
